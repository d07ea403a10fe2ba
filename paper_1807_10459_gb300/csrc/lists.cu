// lists.cu -- per-query sorted neighbour lists in the shared (Y,Z) and Z
// subspaces, the preparation step of ksg_list_kernel (ksg_list.cuh).
//
// For every query i (sorted sample position) and every other sample j that
// may belong to a list, the max-norm distances d_Z(i,j) over the z columns
// and d_YZ(i,j) over the z and y columns of sh are formed exactly as in the
// estimator's definition (fp32 |a-b| and maxima).  List A holds every j != i
// with d_YZ < r_A(i), list B every j != i with d_Z < r_B(i), each ascending
// by distance (equal distances in any order; entries at r itself may follow).
// r_A, r_B are any radii for which the lists fit their capacities.  With
// cap_b = 0 there is only list A.
//
// Two kernels per chunk of queries, with the unsorted entries in scratch
// between them:
//   k_collect     a warp per one or two queries: a radius for each list
//                 from a sample of the distances, then one pass over the
//                 tiles whose box is within a radius, appending the entries.
//   k_sort_lists  a block per (query, list): counting sort on the distance.
// Measured on GB300 against one block per query with two histogram passes over
// all rows and block radix sorts, both kernels together: N = 9995, three z and
// one y column, lists of 2048 and 4096: 1.68 -> 0.77 ms; N = 4997, six z,
// 1024 and 2048: 0.51 -> 0.29 ms; N = 99850, ten z, 512 and 1024: 44.3 ->
// 8.8 ms (that kernel read every visited row once per query, and visited 60 to
// 95 % of the tiles for its histogram).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "ksg_common.cuh"
#include "list_scratch.cuh"

namespace idtx {

namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kBinShift = 19;       // histogram bins: 16 per octave of distance
constexpr int kHistBins = 256;      // 16 octaves
constexpr int kHistPerLane = kHistBins / 32;
constexpr int kCollectWarps = 8;
constexpr int kCollectThreads = kCollectWarps * 32;

// Sampling.  A list's radius is the distance within which 1.15 capacities of
// samples are expected, from a sample holding `hits` of its shorter list's
// entries (a spread of 1 / sqrt(hits)): 64 for lists of 1024 entries or more,
// 28 below, where the sample is a larger share of the work.  A scratch buffer
// takes two capacities, 1.5 from 2048 entries on (their spread is smaller),
// so most lists end full and buffers rarely overflow.
constexpr float kTargetFill = 1.15f;

struct CollectArgs {
    const float *sh;
    int64_t n;
    int64_t q0;          // first query of the chunk
    int n_q;             // queries of the chunk
    int cap_a, cap_b;    // list capacities
    int buf_a, buf_b;    // scratch entries per query
    int n_sample;        // sampled rows (0: no sampling), at `stride`
    int stride;
    int2 *raw_a, *raw_b; // scratch [n_q][buf]
    int4 *raw_meta;      // per query of the chunk: counts, radii (bits)
};

// The radius of a list from a histogram of sampled distances (bin 0 at float
// bits base << 19): the distance below which `want` of them lie, linear
// within its bin; +inf when the histogram's last octave does not reach it.
// Warp-uniform; the lanes hold consecutive bins.
__device__ float hist_radius(const int *hist, int base, float want)
{
    const int lane = threadIdx.x & 31;
    int c[kHistPerLane], sum = 0;
#pragma unroll
    for (int b = 0; b < kHistPerLane; ++b) {
        c[b] = hist[lane * kHistPerLane + b];
        sum += c[b];
    }
    int inc = sum;
    for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(kFull, inc, off);
        if (lane >= off) inc += v;
    }
    const uint32_t over = __ballot_sync(kFull, (float)inc > want);
    float r = INFINITY;
    if (over) {
        const int l = __ffs(over) - 1;
        float mine = 0.0f;
        if (lane == l) {
            int cum = inc - sum;
#pragma unroll
            for (int b = 0; b < kHistPerLane; ++b) {
                if ((float)cum <= want && (float)(cum + c[b]) > want) {
                    const int at = base + l * kHistPerLane + b;
                    const float lo = __uint_as_float((unsigned)max(at, 0) << kBinShift);
                    const float hi = __uint_as_float((unsigned)max(at + 1, 0) << kBinShift);
                    mine = l * kHistPerLane + b == kHistBins - 1
                               ? INFINITY
                               : lo + (hi - lo) * ((want - (float)cum) / (float)c[b]);
                }
                cum += c[b];
            }
        }
        r = __shfl_sync(kFull, mine, l);
    }
    return r;
}

// A full scratch buffer: lower the radius to a bin edge below which at most
// cap entries lie and keep those (in order).  Called by a whole warp.  Every
// sample closer than the new radius that has been met stays listed.
struct Shrunk {
    int kept;
    float radius;
};
__device__ __noinline__ Shrunk shrink_list(int2 *buf, int cnt, int cap, int *hist)
{
    const int lane = threadIdx.x & 31;
    for (int b = lane; b < kHistBins; b += 32) hist[b] = 0;
    unsigned top = 0;
    for (int p = lane; p < cnt; p += 32) top = max(top, (unsigned)buf[p].y);
    top = __reduce_max_sync(kFull, top);
    const int base = (int)(top >> kBinShift) - (kHistBins - 1);
    __syncwarp();
    for (int p = lane; p < cnt; p += 32)
        atomicAdd(&hist[max((int)((unsigned)buf[p].y >> kBinShift) - base, 0)], 1);
    __syncwarp();
    int sum = 0;
    for (int b = 0; b < kHistPerLane; ++b) sum += hist[lane * kHistPerLane + b];
    int inc = sum;
    for (int off = 1; off < 32; off <<= 1) {
        const int v = __shfl_up_sync(kFull, inc, off);
        if (lane >= off) inc += v;
    }
    // the first bin at which the running count exceeds cap (cnt > cap here)
    const int l = __ffs(__ballot_sync(kFull, inc > cap)) - 1;
    int cut = 0;
    if (lane == l) {
        int cum = inc - sum;
        for (int b = 0; b < kHistPerLane; ++b) {
            cum += hist[lane * kHistPerLane + b];
            if (cum > cap) {
                cut = lane * kHistPerLane + b;
                break;
            }
        }
    }
    cut = __shfl_sync(kFull, cut, l);
    // bin 0 also holds what is more than 16 octaves below the largest
    const float radius = cut == 0 ? 0.0f : __uint_as_float((unsigned)max(base + cut, 0) << kBinShift);
    int kept = 0;
    for (int p0 = 0; p0 < cnt; p0 += 32) {
        const int p = p0 + lane;
        const int2 e = p < cnt ? buf[p] : make_int2(0, __float_as_int(INFINITY));
        const bool keep = __int_as_float(e.y) < radius;
        const uint32_t m = __ballot_sync(kFull, keep);  // also orders the reads before the writes
        if (keep) buf[kept + __popc(m & ((1u << lane) - 1u))] = e;
        kept += __popc(m);
        __syncwarp();
    }
    return Shrunk{kept, radius};
}

// One warp per QW (one or two) consecutive queries.
//
// Radii.  The distances to n_sample rows spread evenly over the samples (in
// Morton order, so over space) go into a histogram per list; the radius is
// the distance at the wanted rank of the sample (hist_radius).  It only
// decides how long the lists get: they hold every sample below it.
//
// Tiles.  Rows kTJ and kTJ+1 of every tile of sh hold its samples'
// per-dimension minimum and maximum.  A tile's box gap (the largest over
// dimensions of the distance from the query to the box, 0 inside) bounds its
// samples' distances from below in the definition's fp32 arithmetic (rounding
// is monotone, so the bound holds for the computed distances): tiles whose
// gap reaches both radii of both queries are skipped, 32 tiles being tested
// at a time, one per lane.
//
// A visited tile's rows are loaded once for the warp's queries, whose
// coordinates stay in registers, and the entries below a radius are appended
// to the query's buffers (the counts are the warp's own: no atomics).  With
// more than six dimensions the first four are tested first: a group of 32
// rows none of which is within a radius there goes no further.
// Bound by issue (the differences and maxima) at few dimensions and by L1 at
// many; two queries per warp at 80 registers ran N = 99850, ten z in 7.1 ms,
// four queries at 167 registers (half the warps) in 15.4.
template <int DZ, int DY, int QW>
__global__ void __launch_bounds__(kCollectThreads, QW == 1 ? 4 : (DZ + DY <= 12 ? 3 : 2))
    k_collect(const CollectArgs a)
{
    constexpr int DS = DZ + DY, NC = (DS + 3) / 4, DSP = NC * 4;
    constexpr int kSegs = kTJ / 32;
    constexpr int U = NC == 1 ? 4 : 2;  // rows a lane has in flight
    constexpr bool EARLY = DZ > 6;
    static_assert(kTJ % QW == 0 && kSegs % U == 0, "query groups and row steps tile a tile");
    __shared__ int s_hist[kCollectWarps][QW][2][kHistBins];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g0 = (blockIdx.x * kCollectWarps + warp) * QW;  // first query, within the chunk
    if (g0 >= a.n_q) return;
    const int n = (int)a.n;  // at most IDTX_MAX_N; row offsets in float4 fit an int
    const float4 *sh = reinterpret_cast<const float4 *>(a.sh);
    auto row_of = [&](int j) { return sh + ((j / kTJ) * kTileRows + (j % kTJ)) * NC; };
    auto load = [&](const float4 *p, float(&r)[DSP]) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const float4 v = __ldg(p + c);
            r[4 * c] = v.x, r[4 * c + 1] = v.y, r[4 * c + 2] = v.z, r[4 * c + 3] = v.w;
        }
    };
    auto dist = [](const float(&q)[DSP], const float(&r)[DSP], float &dz, float &dyz) {
        dz = fabsf(q[0] - r[0]);
#pragma unroll
        for (int d = 1; d < DZ; ++d) dz = fmaxf(dz, fabsf(q[d] - r[d]));
        dyz = dz;
#pragma unroll
        for (int d = DZ; d < DS; ++d) dyz = fmaxf(dyz, fabsf(q[d] - r[d]));
    };
    // The second query past the chunk's end (odd counts) repeats the first
    // and lists nothing.
    const bool two = QW > 1 && g0 + 1 < a.n_q;
    const int q0 = (int)a.q0 + g0;
    float q[QW][DSP], ra[QW], rb[QW];
    int ca[QW], cb[QW];
#pragma unroll
    for (int u = 0; u < QW; ++u) {
        load(row_of(q0 + (two ? u : 0)), q[u]);
        ra[u] = rb[u] = INFINITY;
        ca[u] = cb[u] = 0;
    }
    int *hist = s_hist[warp][0][0];
    if (a.n_sample > 0) {
        for (int b = lane; b < QW * 2 * kHistBins; b += 32) hist[b] = 0;
        __syncwarp();
        int base[QW][2];
        for (int s0 = 0; s0 < a.n_sample; s0 += 32) {
            const bool in = s0 + lane < a.n_sample;
            float r[DSP];
            load(row_of(in ? (s0 + lane) * a.stride : 0), r);
#pragma unroll
            for (int u = 0; u < QW; ++u) {
                float dz, dyz;
                dist(q[u], r, dz, dyz);
                const unsigned k[2] = {__float_as_uint(dyz) >> kBinShift, __float_as_uint(dz) >> kBinShift};
#pragma unroll
                for (int l = 0; l < 2; ++l) {
                    // the bins end an octave above the first rows' largest
                    if (s0 == 0) base[u][l] = (int)__reduce_max_sync(kFull, k[l]) + 17 - kHistBins;
                    if (in)
                        atomicAdd(&hist[(u * 2 + l) * kHistBins +
                                        min(max((int)k[l] - base[u][l], 0), kHistBins - 1)], 1);
                }
            }
        }
        __syncwarp();
        const float part = kTargetFill * (float)a.n_sample / (float)n;
#pragma unroll
        for (int u = 0; u < QW; ++u) {
            if (a.cap_a < n - 1)
                ra[u] = hist_radius(hist + u * 2 * kHistBins, base[u][0], part * (float)a.cap_a);
            if (a.cap_b < n - 1)
                rb[u] = hist_radius(hist + (u * 2 + 1) * kHistBins, base[u][1], part * (float)a.cap_b);
        }
        __syncwarp();
    }
#pragma unroll
    for (int u = 0; u < QW; ++u) {
        if (a.cap_b == 0) rb[u] = -1.0f;  // list A only
        if (u > 0 && !two) ra[u] = rb[u] = -1.0f;
    }
    int2 *const oa = a.raw_a + (int64_t)g0 * a.buf_a, *const ob = a.raw_b + (int64_t)g0 * a.buf_b;
    const int n_tiles = (n + kTJ - 1) / kTJ;
    const int home = q0 / kTJ;  // the tile of both queries
    const uint32_t below = (1u << lane) - 1u;
    for (int tb = 0; tb < n_tiles; tb += 32) {
        bool vis = false;
        if (tb + lane < n_tiles) {
            const float4 *bx = sh + ((tb + lane) * kTileRows + kTJ) * NC;
            float lo[DSP], hi[DSP];
            load(bx, lo);
            load(bx + NC, hi);
#pragma unroll
            for (int u = 0; u < QW; ++u) {
                float gz = 0.0f;
#pragma unroll
                for (int d = 0; d < DZ; ++d) gz = fmaxf(gz, fmaxf(lo[d] - q[u][d], q[u][d] - hi[d]));
                float gyz = gz;
#pragma unroll
                for (int d = DZ; d < DS; ++d) gyz = fmaxf(gyz, fmaxf(lo[d] - q[u][d], q[u][d] - hi[d]));
                vis |= gyz < ra[u] || gz < rb[u];
            }
        }
        uint32_t todo = __ballot_sync(kFull, vis);
        while (todo) {
            const int t = tb + __ffs(todo) - 1;
            todo &= todo - 1;
            const float4 *rows = sh + (t * kTileRows + lane) * NC;
            const int self = t == home ? q0 % kTJ : -2;  // the first query's row of this tile
#pragma unroll 1
            for (int s0 = 0; s0 < kSegs; s0 += U) {
                float r[U][DSP];
#pragma unroll
                for (int v = 0; v < U; ++v) load(rows + (s0 + v) * 32 * NC, r[v]);
#pragma unroll
                for (int v = 0; v < U; ++v) {
                    const int at = (s0 + v) * 32 + lane;
#pragma unroll
                    for (int u = 0; u < QW; ++u) {
                        if (EARLY) {
                            float d4 = fabsf(q[u][0] - r[v][0]);
#pragma unroll
                            for (int d = 1; d < 4; ++d) d4 = fmaxf(d4, fabsf(q[u][d] - r[v][d]));
                            if (!__any_sync(kFull, d4 < fmaxf(ra[u], rb[u]))) continue;
                        }
                        float dz, dyz;
                        dist(q[u], r[v], dz, dyz);
                        const bool other = at != self + u;
                        bool pa = dyz < ra[u] && other, pb = dz < rb[u] && other;
                        uint32_t ma = __ballot_sync(kFull, pa), mb = __ballot_sync(kFull, pb);
                        if (ma) {
                            int2 *out = oa + u * a.buf_a;
                            if (ca[u] + __popc(ma) > a.buf_a) {
                                __syncwarp();
                                const Shrunk w = shrink_list(out, ca[u], a.cap_a, hist);
                                ca[u] = w.kept;
                                ra[u] = w.radius;
                                pa = pa && dyz < ra[u];
                                ma = __ballot_sync(kFull, pa);
                            }
                            if (pa) out[ca[u] + __popc(ma & below)] = make_int2(t * kTJ + at, __float_as_int(dyz));
                            ca[u] += __popc(ma);
                        }
                        if (mb) {
                            int2 *out = ob + u * a.buf_b;
                            if (cb[u] + __popc(mb) > a.buf_b) {
                                __syncwarp();
                                const Shrunk w = shrink_list(out, cb[u], a.cap_b, hist);
                                cb[u] = w.kept;
                                rb[u] = w.radius;
                                pb = pb && dz < rb[u];
                                mb = __ballot_sync(kFull, pb);
                            }
                            if (pb) out[cb[u] + __popc(mb & below)] = make_int2(t * kTJ + at, __float_as_int(dz));
                            cb[u] += __popc(mb);
                        }
                    }
                }
            }
        }
    }
    if (lane == 0) {
        a.raw_meta[g0] = make_int4(ca[0], cb[0], __float_as_int(ra[0]), __float_as_int(rb[0]));
        if (two)
            a.raw_meta[g0 + 1] =
                make_int4(ca[QW - 1], cb[QW - 1], __float_as_int(ra[QW - 1]), __float_as_int(rb[QW - 1]));
    }
}

constexpr int kBigBin = 16;  // bins above this are sorted by the whole block
// Bins to sort in place that a block lists (more are found again by a walk over
// all bins).  Short: three blocks of the largest lists take 195.6 of the 196 KB
// that leave the other 60 to L1 (with room for all bins it sorted 6 % slower, as it
// is 3 than without a list).
constexpr int kUnequal = 64;

struct SortArgs {
    const int2 *raw;       // [query of the chunk][buf]
    const int4 *raw_meta;
    int buf, cap;
    int is_b;              // list B's (else list A's) fields of the metas
    int pow;               // squarings of the scaled distance before binning
    int64_t q0;
    int2 *list;
    int4 *meta;
};

struct SortPair {
    SortArgs l[2];
};

// Dynamic shared memory: the bins' offsets, then the entries' keys and samples
// (before them, a copy of the offsets).
__host__ __device__ constexpr size_t sort_smem(int buf, int bins)
{
    const size_t offs = ((size_t)bins + 4) * sizeof(int), ent = (size_t)buf * sizeof(int2);
    return offs + (ent > offs ? ent : offs);
}

// One block per (query, list): the collected entries in ascending order of
// distance, the first `cap` of them written out.  A counting sort over bins
// that are even in a power of the distance (a neighbourhood of dimension D
// holds about r^D samples, so the power evens out the bins).  Where that
// leaves a bin of more than kBigBin entries (a list without a radius, whose
// farthest entries stretch the bins), the bins are refined once; bins that
// are big all the same (many equal distances) are sorted in place by the
// whole block, unless all of their distances are equal.  (All bins were looked
// at in turn and every big one sorted: N = 3000, three z columns of three
// values, lists of 2048 and 3008 entries, 4.0 ms for what is now 0.33.)  The
// other bins hold one or two entries on average and at most
// W + 1; their entries find their places by comparing with the W entries
// before and after them (reads in sequence, no barrier; exchanges of
// neighbours until nothing moves took a third more time: N = 9995, lists of
// 2048 and 4096, 0.74 against 0.57 ms; N = 1000, lists of 512 and 999 without
// a radius, 35 against 27 us, and 68 before bins were refined).
// Bound by instruction issue and shared memory.  T threads, E entries per
// thread, BINS bins.
template <int T, int E, int BINS>
__global__ void __launch_bounds__(T, E > 8 ? 1536 / T : 2048 / T)
    k_sort_lists(const SortPair pair)
{
    constexpr int kWarps = T / 32, nb = BINS;
    extern __shared__ __align__(16) unsigned char s_raw[];
    __shared__ int s_part[kWarps];
    __shared__ unsigned s_top;
    __shared__ int s_most;  // entries of the fullest bin
    __shared__ short s_list[kUnequal];  // bins to sort in place
    __shared__ int s_unequal;           // their number
    const SortArgs &a = pair.l[blockIdx.y];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int qr = blockIdx.x;
    const int64_t i = a.q0 + qr;
    const int cap = a.cap;
    const int2 *raw = a.raw + (int64_t)qr * a.buf;
    int2 *out = a.list + i * cap;
    const int4 rm = a.raw_meta[qr];
    const int n = a.is_b ? rm.y : rm.x;
    const float radius = __int_as_float(a.is_b ? rm.w : rm.z);
    const int sq = a.pow;
    int *base = reinterpret_cast<int *>(s_raw);
    int *keys = base + nb + 4, *vals = keys + a.buf;
    for (int b = tid; b < nb / 4; b += T) reinterpret_cast<int4 *>(base)[b] = make_int4(0, 0, 0, 0);
    if (tid == 0) {
        s_most = 0;
        s_top = 0;
        s_unequal = 0;
    }
    __syncthreads();
    float top = radius;
    if (!(radius < INFINITY)) {  // no radius: the bins span up to the largest distance
        unsigned m = 0;
        for (int p = tid; p < n; p += T) m = max(m, (unsigned)raw[p].y);
        m = __reduce_max_sync(kFull, m);
        if (lane == 0) atomicMax(&s_top, m);
        __syncthreads();
        top = __uint_as_float(s_top);
    }
    const float inv = top > 0.0f ? 1.0f / top : 0.0f, fnb = (float)nb;
    // The entries' bins, counted.  Refined: a second round by the places that
    // a first round's counts give them, each bin's entries spread evenly over
    // its places; its bins are even whatever the distances' distribution.
    // Both are non-decreasing in the distance.
    const int *first = keys;
    const float per_place = fnb / (float)max(n, 1);
    auto bin_of = [&](int key, auto again) {
        float t = __int_as_float(key) * inv;
        if (sq >= 1) t *= t;
        if (sq >= 2) t *= t;
        t *= fnb;
        int b = min(max((int)t, 0), nb - 1);
        if constexpr (decltype(again)::value) {
            const int s0 = first[b], s1 = first[b + 1];
            const float at = fminf((float)s0 + fmaxf(t - (float)b, 0.0f) * (float)(s1 - s0), (float)s1);
            b = min(max((int)(at * per_place), 0), nb - 1);
        }
        return b;
    };
    // The loads of kBatch entries are in flight together (E a multiple of it).
    constexpr int kBatch = E < 8 ? E : (E % 8 == 0 ? 8 : 4);
    static_assert(E % kBatch == 0, "whole batches");
    unsigned at[E];  // bin << 16 | place within the bin (buffers hold under 65536 entries)
    auto count = [&](auto again) {
#pragma unroll
        for (int e0 = 0; e0 < E; e0 += kBatch) {
            if (e0 * T >= n) break;
            int key[kBatch];
#pragma unroll
            for (int e = 0; e < kBatch; ++e) {
                const int p = (e0 + e) * T + tid;
                key[e] = p < n ? raw[p].y : 0;
            }
#pragma unroll
            for (int e = 0; e < kBatch; ++e) {
                const int b = bin_of(key[e], again);
                if ((e0 + e) * T + tid < n)
                    at[e0 + e] = (unsigned)b << 16 | (unsigned)atomicAdd(&base[b], 1);
            }
        }
        __syncthreads();
        // exclusive scan of the bins' counts: a warp takes nb / kWarps
        // consecutive bins, 128 at a time, four a lane
        constexpr int kSteps = nb / (4 * T);
        static_assert(kSteps >= 1, "four bins a thread");
        int4 *mine = reinterpret_cast<int4 *>(base) + warp * kSteps * 32 + lane;
        int4 ex[kSteps];
        int run = 0, most = 0;
#pragma unroll
        for (int b = 0; b < kSteps; ++b) {
            const int4 c = mine[b * 32];
            most = max(most, max(max(c.x, c.y), max(c.z, c.w)));
            const int sum = c.x + c.y + c.z + c.w;
            int inc = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(kFull, inc, o);
                if (lane >= o) inc += v;
            }
            const int x = run + inc - sum;
            ex[b] = make_int4(x, x + c.x, x + c.x + c.y, x + c.x + c.y + c.z);
            run += __shfl_sync(kFull, inc, 31);
        }
        most = __reduce_max_sync(kFull, most);
        if (lane == 0) {
            s_part[warp] = run;
            atomicMax(&s_most, most);
        }
        __syncthreads();
        int before = 0;
        for (int w = 0; w < warp; ++w) before += s_part[w];
#pragma unroll
        for (int b = 0; b < kSteps; ++b)
            mine[b * 32] = make_int4(before + ex[b].x, before + ex[b].y, before + ex[b].z, before + ex[b].w);
        if (tid == 0) base[nb] = n;
        __syncthreads();
    };
    count(std::false_type{});
    if (s_most > kBigBin) {
        for (int b = tid; b <= nb; b += T) {  // the entries are not placed yet
            keys[b] = base[b];
            base[b] = 0;
        }
        __syncthreads();
        if (tid == 0) s_most = 0;
        __syncthreads();
        count(std::true_type{});
    }
#pragma unroll
    for (int e0 = 0; e0 < E; e0 += kBatch) {
        if (e0 * T >= n) break;
        int2 v[kBatch];
#pragma unroll
        for (int e = 0; e < kBatch; ++e) {
            const int p = (e0 + e) * T + tid;
            v[e] = p < n ? raw[p] : make_int2(0, 0);
        }
#pragma unroll
        for (int e = 0; e < kBatch; ++e)
            if ((e0 + e) * T + tid < n) {
                const int p = base[at[e0 + e] >> 16] + (int)(at[e0 + e] & 0xffffu);
                keys[p] = v[e].y;
                vals[p] = v[e].x;
            }
    }
    __syncthreads();
    if (s_most > kBigBin) {
        // The big bins of unequal distances, found by a warp each.
#pragma unroll 1
        for (int b0 = warp * 32; b0 < nb; b0 += T) {
            uint32_t big = __ballot_sync(kFull, base[b0 + lane + 1] - base[b0 + lane] > kBigBin);
            for (; big; big &= big - 1) {
                const int b = b0 + __ffs(big) - 1, s0 = base[b], s1 = base[b + 1];
                int differ = 0;
#pragma unroll 1
                for (int p = s0 + lane; p < s1; p += 32) differ |= keys[p] ^ keys[s0];
                if (__any_sync(kFull, differ) && lane == 0) {
                    const int g = atomicAdd(&s_unequal, 1);
                    if (g < kUnequal) s_list[g] = (short)b;
                }
            }
        }
        __syncthreads();
        // Bitonic sort (ascending-only form, so that any length works: an
        // index past the end counts as +inf and never moves) of each of them,
        // or of every big bin if there are more than the list holds.
        const int n_unequal = s_unequal;
        const bool listed = n_unequal <= kUnequal;
        for (int g = 0; g < (listed ? n_unequal : nb); ++g) {
            const int b = listed ? s_list[g] : g, s0 = base[b], m = base[b + 1] - s0;
            if (m <= kBigBin) continue;
            int half = 1;
            while (2 * half < m) half <<= 1;
            auto exchange = [&](int x, int y) {
                if (y < m) {
                    const int p = keys[s0 + x], r = keys[s0 + y];
                    if (p > r) {
                        keys[s0 + x] = r;
                        keys[s0 + y] = p;
                        const int v = vals[s0 + x];
                        vals[s0 + x] = vals[s0 + y];
                        vals[s0 + y] = v;
                    }
                }
            };
            for (int k = 2; k <= 2 * half; k <<= 1) {
                for (int t = tid; t < half; t += T) {
                    const int blk = t / (k / 2), w = t % (k / 2);
                    exchange(blk * k + w, blk * k + k - 1 - w);
                }
                __syncthreads();
                for (int j = k / 4; j > 0; j >>= 1) {
                    for (int t = tid; t < half; t += T) {
                        const int x = (t / j) * 2 * j + t % j;
                        exchange(x, x + j);
                    }
                    __syncthreads();
                }
            }
        }
    }
    // An entry's place: its own, less the larger ones before it, plus the
    // smaller ones after it (bit patterns of non-negative floats order like
    // integers; equal ones keep their order).  Entries of other bins, and of
    // sorted ones, are on their right side already.
    const int len = min(n, cap), w = min(s_most, kBigBin) - 1;
    for (int p = tid; p < n; p += T) {
        const int key = keys[p];
        int pos = p;
        for (int d = 1; d <= w; ++d) {
            pos -= p >= d && keys[p - d] > key ? 1 : 0;
            pos += p + d < n && keys[p + d] < key ? 1 : 0;
        }
        if (pos < cap) out[pos] = make_int2(vals[p], key);
        if (pos == cap) {  // a cut list's radius is its first dropped distance
            if (a.is_b)
                a.meta[i].w = key;
            else
                a.meta[i].z = key;
        }
    }
    const int end = min(cap, (n + 31) & ~31);
    for (int p = n + tid; p < end; p += T) out[p] = make_int2(0, __float_as_int(INFINITY));
    if (tid == 0) {
        if (a.is_b) {
            a.meta[i].y = len;
            if (n <= cap) a.meta[i].w = __float_as_int(radius);
        } else {
            a.meta[i].x = len;
            if (n <= cap) a.meta[i].z = __float_as_int(radius);
        }
    }
}

// Two queries a warp share a visited tile's rows, one leaves more registers for
// warps (four blocks an SM instead of three) and twice the warps: better as long
// as the rows stay in L1 and are short, and for few queries.  One against two,
// us: N = 1000, two z, 11 and 17; 2500, eight, 39 and 49; 4997, six, 86 and
// 100; 9995, three, 205 and 269; 30000, three, 513 and 610; 50000, two, 736 and
// 706; 4000, eight, 88 (at three blocks) and 73; 30000, eight, 1705 and 1469.
template <int DZ, int DY>
constexpr int kCollectSingle = DZ + DY <= 8 ? 32768 : 2560;
template <int DZ, int DY>
cudaError_t launch_collect(const CollectArgs &a, cudaStream_t st)
{
    if (a.n <= kCollectSingle<DZ, DY>)
        k_collect<DZ, DY, 1><<<(unsigned)((a.n_q + kCollectWarps - 1) / kCollectWarps), kCollectThreads,
                               0, st>>>(a);
    else
        k_collect<DZ, DY, 2><<<(unsigned)((a.n_q + 2 * kCollectWarps - 1) / (2 * kCollectWarps)),
                               kCollectThreads, 0, st>>>(a);
    return cudaGetLastError();
}

template <int DY>
cudaError_t collect_dz(int dzb, const CollectArgs &a, cudaStream_t st)
{
    switch (dzb) {
    case 1: return launch_collect<1, DY>(a, st);
    case 2: return launch_collect<2, DY>(a, st);
    case 3: return launch_collect<3, DY>(a, st);
    case 4: return launch_collect<4, DY>(a, st);
    case 5: return launch_collect<5, DY>(a, st);
    case 6: return launch_collect<6, DY>(a, st);
    case 8: return launch_collect<8, DY>(a, st);
    case 10: return launch_collect<10, DY>(a, st);
    case 12: return launch_collect<12, DY>(a, st);
    case 16: return launch_collect<16, DY>(a, st);
    default: return cudaErrorInvalidValue;
    }
}

template <int T, int E, int BINS>
cudaError_t launch_sort(const SortPair &p, int n_q, int lists, int buf, cudaStream_t st)
{
    static DeviceOnce attr;  // the attribute is per function and device
    cudaError_t e = once_per_device(attr, [&](int) {
        return cudaFuncSetAttribute(k_sort_lists<T, E, BINS>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)sort_smem(E * T, BINS));
    });
    if (e != cudaSuccess || n_q <= 0) return e;
    k_sort_lists<T, E, BINS>
        <<<dim3((unsigned)n_q, (unsigned)lists), T, sort_smem(buf, BINS), st>>>(p);
    return cudaGetLastError();
}

// Lists of `buf` scratch entries (n_q = 0: set-up only).  Threads per block
// by the buffer, so that a thread has at most 12 entries and the SM's threads
// are full or nearly so.
cudaError_t sort_lists(const SortPair &p, int n_q, int lists, int buf, cudaStream_t st)
{
    if (buf <= 512) return launch_sort<128, 4, 512>(p, n_q, lists, buf, st);
    if (buf <= 1024) return launch_sort<128, 8, 1024>(p, n_q, lists, buf, st);
    if (buf <= 2048) return launch_sort<256, 8, 2048>(p, n_q, lists, buf, st);
    if (buf <= 4096) return launch_sort<512, 8, 4096>(p, n_q, lists, buf, st);
    return launch_sort<512, 12, 4096>(p, n_q, lists, buf, st);
}

static_assert(kMaxListB + kMaxListB / 2 <= 512 * 12, "the largest buffer");
static_assert(kScratchTile == kTJ && kListEntry == sizeof(int2) && kListMeta == sizeof(int4), "list_scratch.cuh");

}  // namespace

cudaError_t build_lists(const float *sh, int dzb, int dyb, int dz, int dy, int64_t n, int cap_a, int cap_b,
                        int2 *list_a, int2 *list_b, int4 *meta, void *scratch, cudaStream_t st,
                        int *launches)
{
    if (launches) *launches = 0;
    if (n <= 0) {  // set-up only: every instantiation's attribute (outside captures)
        cudaError_t e = cudaSuccess;
        for (int buf = 512; buf <= 8192 && e == cudaSuccess; buf *= 2)
            e = sort_lists(SortPair{}, 0, 0, buf, st);
        return e;
    }
    const int64_t chunk = chunk_of(n, cap_a, cap_b);
    CollectArgs c{};
    c.sh = sh;
    c.n = n;
    c.cap_a = cap_a;
    c.cap_b = cap_b;
    c.buf_a = buf_of(cap_a, n);
    c.buf_b = buf_of(cap_b, n);
    c.raw_a = (int2 *)scratch;
    c.raw_b = c.raw_a + chunk * c.buf_a;
    c.raw_meta = (int4 *)(((uintptr_t)(c.raw_b + chunk * c.buf_b) + 15) & ~(uintptr_t)15);
    // No sample when it would be half of the samples or every list holds all.
    const int cut = cap_a < n - 1 || cap_b == 0 ? cap_a : cap_b;
    if (cut < n - 1) {
        const int64_t m = (cut >= 1024 ? 64 : 28) * n / cut;
        if (2 * m <= n) {
            c.stride = (int)(n / m);
            c.n_sample = (int)((n + c.stride - 1) / c.stride);
        }
    }
    // squarings: the power of the distance that evens out the bins, by the true
    // dimensions (the buckets' other columns are zero: with their number the
    // widest specialisation's bins of two z columns were by far too uneven;
    // N = 3000, lists of 2048 and 3008 entries, 959 us against 178)
    auto squarings = [](int d) { return d >= 4 ? 2 : (d >= 2 ? 1 : 0); };
    SortPair s{};
    s.l[0] = SortArgs{c.raw_a, c.raw_meta, c.buf_a, cap_a, 0, squarings(dz + dy), 0, list_a, meta};
    s.l[1] = SortArgs{c.raw_b, c.raw_meta, c.buf_b, cap_b, 1, squarings(dz), 0, list_b, meta};
    for (int64_t q0 = 0; q0 < n; q0 += chunk) {
        const int n_q = (int)std::min(chunk, n - q0);
        c.q0 = s.l[0].q0 = s.l[1].q0 = q0;
        c.n_q = n_q;
        cudaError_t e = dyb == 1   ? collect_dz<1>(dzb, c, st)
                        : dyb == 2 ? collect_dz<2>(dzb, c, st)
                        : dyb == 4 && dzb == 16 ? launch_collect<16, 4>(c, st)
                                                : cudaErrorInvalidValue;
        if (e != cudaSuccess) return e;
        // Short lists in one launch; long ones apart, with the blocks of each size.
        const int buf = std::max(c.buf_a, c.buf_b);
        const bool together = cap_b > 0 && (buf <= 1024 || c.buf_a == c.buf_b);
        e = sort_lists(s, n_q, together ? 2 : 1, together ? buf : c.buf_a, st);
        if (e == cudaSuccess && !together && cap_b > 0)
            e = sort_lists(SortPair{{s.l[1], s.l[1]}}, n_q, 1, c.buf_b, st);
        if (e != cudaSuccess) return e;
        if (launches) *launches += together || cap_b == 0 ? 2 : 3;
    }
    return cudaSuccess;
}

}  // namespace idtx
