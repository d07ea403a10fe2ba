// ksg_list.cuh -- the KSG estimator over per-query sorted neighbour lists.
//
// Computes the same statistics as ksg_fused_kernel (ksg_kernel.cuh) -- for
// every job g of a group and every query sample i, eps_i (k-th smallest
// max-norm distance to j != i in (X_g, Y, Z)), the strict-radius counts n_xz,
// n_yz, n_z and the digamma term (KSG algorithm 1, conditional form, the
// estimator named in the IDTxl paper's Summary) -- in another order of work.
//
// Every job of a group shares Y and Z (a surrogate only permutes X; the
// candidates of one greedy step differ only in X), so the neighbourhoods in
// the (Y,Z) and Z subspaces are the same for all of them.  build_lists
// (lists.cu) lists them once per query i, for all jobs together:
//   list A: every j != i with d_YZ(i,j) < r_A(i), ascending by d_YZ,
//   list B: every j != i with d_Z(i,j)  < r_B(i), ascending by d_Z,
// at most cap_a / cap_b entries, r_A and r_B chosen so.  Per (query, job):
//   pass A: eps_i = k-th smallest of max(d_X, d_YZ) over j != i.  Walking
//     list A in order, an entry whose d_YZ is at least the current k-th value
//     cannot enter (the joint distance is at least d_YZ), nor can any later
//     one, so the walk stops there.  If the list runs out while the k-th
//     value is still above r_A, an unlisted sample might enter: that job is
//     recomputed by a full scan.
//   pass B: n_yz = #{list A entries with d_YZ < eps} (bisection of the prefix
//     pass A walked); n_z and n_xz counted over the list B entries with
//     d_Z < eps, using max(d_X, d_Z) < eps <=> d_X < eps and d_Z < eps.  Both
//     are exact when eps <= r_A and eps <= r_B (every sample closer than eps
//     is listed); otherwise the job's counts come from a full scan.
// Every distance is formed from the same fp32 differences and maxima as in
// the definition, so eps and the counts are exact, and a query tile's digamma
// terms are summed without rounding (kPsiBits), as by ksg_fused_kernel: both
// kernels give bit-identical estimates and either may serve a call.
//
// Design (GB300).  The kernel is persistent: one CTA of 32 warps per SM, one
// job per lane.  A CTA takes chunks of consecutive queries of one job group
// (chunks ordered query block by query block, so the CTAs in flight share the
// lists of one block of queries), and its warps take the chunk's queries one
// at a time.  So at any moment the SM's warps serve ~32 consecutive queries of
// one group: samples are in Morton order of (Z, Y), the neighbourhoods of
// consecutive queries overlap, and the X rows the walks gather (one 128-byte
// row of xi per list entry: the 32 jobs' X at that sample) are reused from L1
// instead of L2.
//   * Walks stage their list 32 entries at a time into the warp's buffer and
//     fetch the X rows of the next IDTX_LIST_SA entries while they use those
//     of the last.  The shared walks are warp-uniform (they stop when every
//     lane's job is done); the one or two jobs that would lengthen the
//     neighbour walk most finish lane-split (the 32 lanes splitting the
//     entries), the last of the count walk with the lanes shared out among
//     them.
//   * The counts go out (16 bits each, 32 above 65536 samples) and sum_terms
//     (sums.cu) forms and sums the terms.  No order of the queries matters, so
//     the CTAs take chunks as they come free; (query, group)s that need full
//     scans are queued for ksg_scan_kernel.  Waits (for a chunk being fetched)
//     are bounded by %globaltimer; on expiry the CTA records kErrTimeout and
//     stops.
//   * Calls of at most one z column (n_pad <= 65536) walk an order instead of a
//     list where the subspace has one dimension: with one z column the samples
//     are ordered by it, and the samples after and before the query, whose d_Z
//     ascends, are list B (up to thousands of entries there, beyond any list's
//     capacity); with none and one y column the order is by y and stands for
//     list A.  Without z, n_z is all and n_xz with one x column is a range of
//     the sorted column.  The call, by the tile kernel and so: N = 3001, no z,
//     201 estimates, 1.93 and 0.32 ms; N = 20000, 48.5 and 2.2; one z, N = 3001,
//     0.65 and 0.50 (0.95 with a list B); N = 50000, 101 estimates, 23.1 and 11.5
//     (on data of few values the tile kernel is up to a tenth slower in this
//     order than along a Morton curve, on continuous data faster by up to two
//     thirds).
// Measured on GB300, greedy step of N = 9995 with 9447 estimates (one network;
// lists of 2048 and 4096), against summing the terms in the kernel and scanning
// in place: 19.1 -> 12.7 ms; of N = 4997, six conditions, 28341 estimates: 10.8
// -> 8.5 ms; N = 1000, 101 estimates: 163 -> 24 us (each with sum_terms' 0.27,
// 0.38 ms and 4 us to add).  Bound by issue (71 % of the slots in a capture of 752
// estimates) and L1 (80 % of its rate): fewer, fatter warps (24 of 80 registers)
// were 8 % slower.
#pragma once

#include <type_traits>

#include "ksg_kernel.cuh"
#include "ksg_plain.cuh"

// List entries whose X rows a walk has in flight (4, 8 or 16: whole steps of the
// 32 entries staged at a time; compile-time knobs, the defaults are the tuned
// values).  N = 9995, three z, 2001 estimates, the kernel: 2.96 / 2.84 / 3.15 ms.
#ifndef IDTX_LIST_SA
#define IDTX_LIST_SA 8
#endif
// Jobs of a warp whose neighbour walk goes on past the others' and is finished
// with the lanes splitting its entries (1 / 2 / 3 / 4: 2.89 / 2.84 / 2.86 / 2.92).
#ifndef IDTX_LIST_TAIL_A
#define IDTX_LIST_TAIL_A 2
#endif
// The shared count walk hands over to the repacked phases once at most this
// many jobs (a power of two <= 16) still need entries (4 / 8 / 16: 2.95 / 2.84 /
// 2.87).
#ifndef IDTX_LIST_REPACK
#define IDTX_LIST_REPACK 8
#endif
// Entries a lane takes per step of a repacked count phase (their loads are in
// flight together; entries past the lane's job are predicated off); four with
// more than one x column.  N = 9995, three z, 2001 estimates, the kernel at 2 /
// 4 / 5 / 6 / 8: 2.91 / 2.84 / 2.82 / 2.80 / 2.86 ms.
#ifndef IDTX_LIST_PHASE_STEP
#define IDTX_LIST_PHASE_STEP 6
#endif
// Job groups per super-block of the chunk order (see the kernel).
#ifndef IDTX_LIST_GSB
#define IDTX_LIST_GSB 16
#endif
// Most consecutive queries a CTA takes at a time (256 to 1024 are alike).
#ifndef IDTX_LIST_CHUNKQ
#define IDTX_LIST_CHUNKQ 256
#endif

namespace idtx {

// Number of the ascending distances dist(0..hi-1) (hi the lane's own) that
// are below v, for every lane of a warp.  Warp-uniform probes of every lane
// at once first bound the answers by a power of two (most are far below hi);
// then each lane bisects without branches.
template <typename Dist>
__device__ __forceinline__ int count_below(int hi, float v, Dist dist)
{
    constexpr unsigned kFull = 0xffffffffu;
    int bits = 4;  // the answers are below 2^bits
    while (__any_sync(kFull, (1 << bits) <= hi && dist((1 << bits) - 1) < v)) ++bits;
    int lo = 0;
    for (int b = (1 << bits) >> 1; b; b >>= 1)
        if (lo + b <= hi && dist(lo + b - 1) < v) lo += b;
    return lo;
}

// Number of samples other than the query's own within eps of x in the
// ascending column xs[0..n), which holds x itself: fl(|x - v|) is monotone on
// either side of x, so they are a contiguous range.
__device__ __forceinline__ int count_sorted(const float *xs, int n, float x, float eps)
{
    int top = 1;
    while (2 * top <= n) top <<= 1;
    int lo = 0, hi = 0;  // entries before the range, entries up to its end
    for (int b = top; b; b >>= 1) {
        if (lo + b <= n) {
            const float v = __ldg(xs + lo + b - 1);
            if (v < x && fabsf(x - v) >= eps) lo += b;
        }
        if (hi + b <= n) {
            const float v = __ldg(xs + hi + b - 1);
            if (!(v > x && fabsf(x - v) >= eps)) hi += b;
        }
    }
    return eps > 0.0f ? hi - lo - 1 : 0;
}

// The X values of a job at a sample, in one load (they are aligned to their
// size).  As DX single loads they touched every line of a row DX times; list
// kernel: dx = 3, N = 1000, 101 estimates, 122 -> 85 us; dx = 4, N = 10000, 201,
// 12.7 -> 6.3 ms; dx = 2, N = 10000, 101, three z columns 361 -> 273 us.
template <int DX>
__device__ __forceinline__ void load_x(const float *p, float (&r)[DX])
{
    if constexpr (DX == 4) {
        const float4 v = *reinterpret_cast<const float4 *>(p);
        r[0] = v.x, r[1] = v.y, r[2] = v.z, r[3] = v.w;
    } else if constexpr (DX == 2) {
        const float2 v = *reinterpret_cast<const float2 *>(p);
        r[0] = v.x, r[1] = v.y;
    } else {
#pragma unroll
        for (int d = 0; d < DX; ++d) r[d] = p[d];
    }
}

// Warp minimum / maximum of non-negative floats (distances, +inf allowed):
// their bit patterns order like unsigned integers, so one redux does it.
__device__ __forceinline__ float warp_min_nn(float v)
{
    return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v)));
}

__device__ __forceinline__ float warp_max_nn(float v)
{
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

// Launch shape of the list kernel for one specialisation.  QC: the tile
// kernel's queries per CTA: sum_terms writes one partial sum per QC queries.
template <int DX, int DY, int DZ, int K1, bool EXACT, int QCTA, int NWARPS>
struct ListShape {
    using S = KsgShape<DX, DY, DZ, K1, EXACT, QCTA, NWARPS>;
    static constexpr int QC = S::QC;
    // 32 warps (64 registers a thread) for the small specialisations; 16
    // warps give the wide runtime-k one 128 registers.
    static constexpr int NW = (DX > 2 || K1 > 8) ? 16 : 32;
    static constexpr int THREADS = NW * 32;
    static_assert(QC <= 64, "sum_terms takes tiles of up to 64 queries");
    struct Smem {
        int2 ent[NW][64];  // per warp: two chunks of staged list entries
        unsigned long long work[NW][kNumWork];
        // the CTA's chunks in their order (number, chunk; a ring), the next query
        // (number << 16 | query within the chunk), and the chunk to follow (-1:
        // being fetched)
        int2 chunk[8];
        unsigned cur;
        int ahead;
    };
    static constexpr size_t SMEM = sizeof(Smem);
};

// (query, group)s with full scans for at most this many jobs, and for more,
// are queued apart, from the two ends of KsgLaunch::scans (ksg_scan_kernel).
constexpr int kFewJobs = 8;

// Merge four distances into the ascending h[0..4): sort them, take the four
// smallest of both (the element-wise minimum of one and the other reversed),
// and order that bitonic sequence.  22 minima and maxima without a branch,
// against 28 for four insertions; in a warp of 32 jobs nearly every group of
// four holds a distance for some job's h, so skipping it rarely pays.
__device__ __forceinline__ void cmp_swap(float &a, float &b)
{
    const float lo = fminf(a, b);
    b = fmaxf(a, b);
    a = lo;
}
__device__ __forceinline__ void merge4(float (&h)[4], float s0, float s1, float s2, float s3)
{
    cmp_swap(s0, s1);
    cmp_swap(s2, s3);
    cmp_swap(s0, s2);
    cmp_swap(s1, s3);
    cmp_swap(s1, s2);
    h[0] = fminf(h[0], s3);
    h[1] = fminf(h[1], s2);
    h[2] = fminf(h[2], s1);
    h[3] = fminf(h[3], s0);
    cmp_swap(h[0], h[2]);
    cmp_swap(h[1], h[3]);
    cmp_swap(h[0], h[1]);
    cmp_swap(h[2], h[3]);
}

template <int DX, int DY, int DZ, int K1, bool EXACT, int QCTA, int NWARPS>
__global__ void __launch_bounds__(ListShape<DX, DY, DZ, K1, EXACT, QCTA, NWARPS>::THREADS, 1)
    ksg_list_kernel(const KsgLaunch a, const int n_groups, const int n_chunks, const int chunk_q)
{
    using S = KsgShape<DX, DY, DZ, K1, EXACT, QCTA, NWARPS>;
    using LS = ListShape<DX, DY, DZ, K1, EXACT, QCTA, NWARPS>;
    constexpr int DSP = S::DSP, XW = S::XW, GB = S::GB;
    constexpr int NW = LS::NW;
    constexpr int KH = K1 - 1;  // smallest distances kept (EXACT: exactly k)
    constexpr int kShStage = kTileRows * DSP;
    constexpr unsigned kFull = 0xffffffffu;
    // may serve calls of at most one z column: the generic one covers any dz
    constexpr bool LOW = DZ == 1 || K1 > 8;
    // One z column: n_z is in the thousands, and is found by bisection after the
    // walk for n_xz, not counted in it (which also spilled 32 bytes, now 8).  N =
    // 9995, 9045 estimates, 59.1 -> 56.2 ms; N = 1000, 1001 estimates, 177 -> 182
    // us, and for a runtime k 135 -> 142, with nothing gained at N = 10000.
    constexpr bool SEARCH_Z = DZ == 1 && EXACT;
    constexpr int TAIL_A = IDTX_LIST_TAIL_A;  // jobs left after the shared neighbour walk
    const float kInf = CUDART_INF_F;

    extern __shared__ __align__(16) unsigned char l_smem[];
    auto &sm = *reinterpret_cast<typename LS::Smem *>(l_smem);

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    if (tid == 0) {
        sm.cur = 0;
        sm.chunk[0] = make_int2(0, atomicAdd(a.next, 1));
        sm.ahead = atomicAdd(a.next, 1);
    }
    __syncthreads();

    int2 *ent = sm.ent[warp];
    const int2 sentinel = make_int2(0, __float_as_int(CUDART_INF_F));
    const int kk = a.k;
    auto kth = [&](const float(&h)[KH]) { return EXACT ? h[KH - 1] : select_kth<KH>(h, kk - 1); };
    auto sh_row = [&](int64_t j) { return a.sh + (j / kTJ) * kShStage + (j % kTJ) * DSP; };
    const long long t_begin = clock64();
    unsigned long long my_work = 0;   // work counter `lane` of this warp (5: cycles)
    int grp = 0, num_of = -1, q_of = 0;  // the last query's group and chunk

    while (true) {
        // ---------------- take the CTA's next query.  Chunks of consecutive
        // queries of one group run in super-blocks of GSB groups, query block
        // by query block within a super-block, so the CTAs in flight share a
        // few groups' X rows and a range of queries' lists in L2, while each
        // CTA's warps serve consecutive queries of one group.
        // Chunks of `chunk_q` queries, taken by the CTAs as they come free
        // (the queries' work differs).  The warp that takes the first
        // query past a chunk brings in the one fetched ahead; others that
        // come before it has try again.
        unsigned v = 0;
        if (lane == 0) v = atomicAdd(&sm.cur, 1u);
        v = __shfl_sync(kFull, v, 0);
        const int num = static_cast<int>(v >> 16), at = static_cast<int>(v & 0xffffu);
        if (at >= chunk_q) {
            int ok = 1;
            if (lane == 0) {
                const long long t0 = global_ns();
                if (at == chunk_q) {
                    volatile int *ahead = &sm.ahead;
                    while (ok && *ahead < 0) {
                        __nanosleep(32);
                        ok = global_ns() - t0 <= a.timeout_ns;
                    }
                    if (ok) {
                        const int next = *ahead;
                        *ahead = -1;
                        sm.chunk[(num + 1) & 7] = make_int2((num + 1) & 0xffff, next);
                        __threadfence_block();
                        atomicExch(&sm.cur, static_cast<unsigned>(num + 1) << 16);
                        *ahead = next < n_chunks ? atomicAdd(a.next, 1) : next;
                    }
                } else {
                    const volatile unsigned *cur = &sm.cur;
                    while (ok && (*cur >> 16) == (v >> 16)) {
                        __nanosleep(32);
                        ok = global_ns() - t0 <= a.timeout_ns;
                    }
                }
            }
            if (!__shfl_sync(kFull, ok, 0)) {
                if (lane == 0) atomicOr(a.err, kErrTimeout);
                break;
            }
            continue;
        }
        if (num != num_of) {
            num_of = num;
            __threadfence_block();
            const int2 mine = sm.chunk[num & 7];
            if (mine.x != num) {  // overtaken by seven chunks: cannot be, and is not passed over
                if (lane == 0) atomicOr(a.err, kErrInternal);
                break;
            }
            const int chunk = mine.y;
            if (chunk >= n_chunks) break;
            const int n_qb = (static_cast<int>(a.n) + chunk_q - 1) / chunk_q;
            const int per_sb = IDTX_LIST_GSB * n_qb;
            const int sb = chunk / per_sb;
            const int g0 = sb * IDTX_LIST_GSB;
            const int gs = n_groups - g0 < IDTX_LIST_GSB ? n_groups - g0 : IDTX_LIST_GSB;
            const int rc = chunk - sb * per_sb;
            const int qblock = rc / gs;
            grp = g0 + (rc - qblock * gs);
            q_of = qblock * chunk_q;
        }
        const int qi = q_of + at;  // the query (sorted position)
        const int job = grp * GB + lane;
        const bool job_ok = job < a.n_jobs;

        if (qi < a.n) {
            const float *xg = a.xi + static_cast<int64_t>(grp) * a.n_pad * XW + lane * DX;
            // per-query work counters (warp-uniform)
            unsigned ta = 0, tb = 0, nfa = 0, nfb = 0;
            float xq[DX];
            load_x<DX>(xg + static_cast<int64_t>(qi) * XW, xq);
            // Where a walk's entries come from: a list, or (dir 1 / -1) the
            // samples after / before the query in an order sorted by column
            // `col` of sh, which ascend in their distance in that column.
            struct Src {
                const int2 *l;
                int len, dir, col;
            };
            auto entry = [&](const Src &src, int e) -> int2 {
                if (e >= src.len) return sentinel;
                if (!LOW || src.dir == 0) return __ldg(src.l + e);
                const int j = qi + src.dir * (1 + e);
                return make_int2(j, __float_as_int(fabsf(sh_row(qi)[src.col] - sh_row(j)[src.col])));
            };
            auto entry_d = [&](const Src &src, int e) {  // its distance, e < src.len
                if (!LOW || src.dir == 0) return __int_as_float(__ldg(&src.l[e].y));
                return fabsf(sh_row(qi)[src.col] - sh_row(qi + src.dir * (1 + e))[src.col]);
            };
            // the samples on one side of the query in the order by column col
            auto side = [&](int dir, int col) {
                return Src{nullptr, dir > 0 ? static_cast<int>(a.n) - 1 - qi : qi, dir, col};
            };
            const bool iv_a = LOW && a.iv_a;  // pass A over the order by the y column
            Src la;
            if (iv_a) {
                la = side(1, DZ);
            } else {
                la = Src{a.list_a + static_cast<int64_t>(qi) * a.cap_a, __ldg(&a.lmeta[qi].x), 0, 0};
            }

            // ---------------- pass A: the k smallest joint distances
            float h[KH];
#pragma unroll
            for (int t = 0; t < KH; ++t) h[t] = kInf;
            float th = job_ok ? kInf : -1.0f;  // padding jobs never insert
            int walked_a = 0;
            uint32_t amask = 0;  // jobs the shared walk left to finish lane-split
            // A walk's next rows, fetched while the current ones are used: the
            // entries of list l from e on (staged 32 at a time into the half
            // of the warp's buffer that was used up; past the list's end
            // sentinels), their distances and X values.
            constexpr int SW = IDTX_LIST_SA;
            static_assert(SW % 4 == 0 && 32 % SW == 0, "steps stay within the staged entries");
            float row_d[SW], row_x[SW][DX];
            int2 nxt;
            auto fetch = [&](int e) {
#pragma unroll
                for (int t = 0; t < SW; t += 2) {
                    const int4 v = *reinterpret_cast<const int4 *>(&ent[(e & 63) + t]);
                    row_d[t] = __int_as_float(v.y);
                    row_d[t + 1] = __int_as_float(v.w);
                    // (32 x 32 -> 64 bits: one multiply-add per row)
                    const float *x0 = xg + static_cast<uint64_t>(static_cast<uint32_t>(v.x)) * XW;
                    const float *x1 = xg + static_cast<uint64_t>(static_cast<uint32_t>(v.z)) * XW;
                    load_x<DX>(x0, row_x[t]);
                    load_x<DX>(x1, row_x[t + 1]);
                }
            };
            auto begin = [&](const Src &src) {
                const int2 first = entry(src, lane);
                nxt = entry(src, 32 + lane);
                __syncwarp();
                ent[lane] = first;
                __syncwarp();
                fetch(0);
            };
            auto advance = [&](const Src &src, int e) {  // after the rows of e
                if ((e & 31) == 32 - 2 * SW || (SW > 8 && (e & 31) == 0)) {
                    const int at = (e & ~31) + 32;  // the chunk after e's
                    __syncwarp();
                    ent[(at & 32) + lane] = nxt;
                    __syncwarp();
                    nxt = entry(src, at + 32 + lane);
                }
                fetch(e + SW);
            };
            int my_walked = 0, up_walked = 0;
            const int parts_a = iv_a ? 2 : 1;
            int walk_total = 0;
#pragma unroll 1
            for (int part = 0; part < parts_a; ++part) {
                if (part) {  // then the samples before the query
                    up_walked = my_walked;
                    la = side(-1, DZ);
                }
                begin(la);
                for (int e = 0;; e += SW) {
                    // Ascending list: once the first of the next entries is out
                    // of a job's reach, so is everything after it.  When at most
                    // TAIL_A jobs are still in reach the shared walk stops and
                    // those finish lane-split below.
                    const uint32_t act = __ballot_sync(kFull, row_d[0] < th);
                    if (__popc(act) <= TAIL_A) {
                        amask = act;
                        walked_a = e;
                        break;
                    }
                    float dd[SW];
#pragma unroll
                    for (int t = 0; t < SW; ++t) {
                        float dx = fabsf(xq[0] - row_x[t][0]);
#pragma unroll
                        for (int d = 1; d < DX; ++d) dx = fmaxf(dx, fabsf(xq[d] - row_x[t][d]));
                        dd[t] = fmaxf(dx, row_d[t]);
                    }
                    advance(la, e);
                    if constexpr (EXACT && KH == 4) {
#pragma unroll
                        for (int t = 0; t < SW; t += 4) merge4(h, dd[t], dd[t + 1], dd[t + 2], dd[t + 3]);
                        if (job_ok) th = h[3];
                    } else {
#pragma unroll
                        for (int t = 0; t < SW; ++t) {
                            if (dd[t] < th) {
                                sorted_insert<KH>(h, dd[t]);
                                th = kth(h);
                            }
                        }
                    }
                }
                if (walked_a > la.len) walked_a = la.len;
                // Lane-split finish of the remaining jobs, one at a time: steps of
                // two blocks of 32 entries, one entry per lane and block; the
                // distances below the job's k-th value are inserted smallest first
                // (warp minimum) into its k smallest, which every lane holds,
                // until the step's last entry is out of reach.
                // my_walked: the prefix of list A this lane's job walked.
                my_walked = walked_a;
                while (amask) {
                    const int f = __ffs(amask) - 1;
                    amask &= amask - 1;
                    float xf[DX];
#pragma unroll
                    for (int d = 0; d < DX; ++d) xf[d] = __shfl_sync(kFull, xq[d], f);
                    const float *xgf = xg - lane * DX + f * DX;
                    float hf[KH];
#pragma unroll
                    for (int t = 0; t < KH; ++t) hf[t] = __shfl_sync(kFull, h[t], f);
                    float thf = kth(hf);
                    int pos = walked_a;
                    while (pos < la.len) {
                        const int2 e0 = entry(la, pos + lane), e1 = entry(la, pos + 32 + lane);
                        const float y0 = __int_as_float(e0.y), y1 = __int_as_float(e1.y);
                        if (!(__shfl_sync(kFull, y0, 0) < thf)) break;
                        auto reach = [&](const int2 e, float y) {  // joint distance, +inf out of reach
                            if (!(y < thf)) return kInf;
                            float xr[DX];
                            load_x<DX>(xgf + static_cast<uint64_t>(static_cast<uint32_t>(e.x)) * XW, xr);
                            float dx = fabsf(xf[0] - xr[0]);
#pragma unroll
                            for (int d = 1; d < DX; ++d) dx = fmaxf(dx, fabsf(xf[d] - xr[d]));
                            return fmaxf(dx, y);
                        };
                        float c0 = reach(e0, y0), c1 = reach(e1, y1);
                        while (true) {
                            const float mn = warp_min_nn(fminf(c0, c1));
                            if (!(mn < thf)) break;
                            const uint32_t w0 = __ballot_sync(kFull, c0 == mn);
                            if (w0) {
                                if (lane == __ffs(w0) - 1) c0 = kInf;
                            } else {
                                const uint32_t w1 = __ballot_sync(kFull, c1 == mn);
                                if (lane == __ffs(w1) - 1) c1 = kInf;
                            }
                            sorted_insert<KH>(hf, mn);
                            thf = kth(hf);
                        }
                        ta += (la.len - pos < 64) ? static_cast<unsigned>(la.len - pos) : 64u;
                        pos += 64;
                        // ascending: if the step's last entry is out of reach, so is the rest
                        if (!(__shfl_sync(kFull, y1, 31) < thf)) break;
                    }
                    if (lane == f) {
#pragma unroll
                        for (int t = 0; t < KH; ++t) h[t] = hf[t];
                        th = thf;
                        my_walked = pos < la.len ? pos : la.len;
                    }
                }
                walk_total += walked_a;
            }
            walked_a = walk_total;
            // The list ran out before the job's k-th distance dropped to r_A: eps
            // is sought over every sample (ksg_scan_kernel).
            const float r_a = iv_a ? kInf : __int_as_float(__ldg(&a.lmeta[qi].z));
            const bool fa = job_ok && th > r_a;
            nfa = __popc(__ballot_sync(kFull, fa));
            const float eps = job_ok ? kth(h) : -1.0f;

            // ---------------- pass B: strict-radius counts
            const int b_form = LOW ? a.b_form : 0;
            const float r_b = b_form ? kInf : __int_as_float(__ldg(&a.lmeta[qi].w));
            const bool fb = fa || (job_ok && (eps > r_a || eps > r_b));
            int nz = 0, nyz = 0, nxz = 0;
            // Every list A entry below eps lies in the walked prefix (the walk
            // went on until each job's k-th value was at most the next entry).
            nyz = count_below(job_ok && !fb ? my_walked : 0, eps, [&](int e) { return entry_d(la, e); });
            if (iv_a) {
                const Src up = side(1, DZ);
                nyz += count_below(job_ok && !fb ? up_walked : 0, eps, [&](int e) { return entry_d(up, e); });
            }
            // The count walk over list B: for every job the entries below its
            // eps (n_z) and those also within eps in X (n_xz).  Shared rows,
            // one job per lane, while more than IDTX_LIST_REPACK jobs need
            // entries (`reach`: a job's eps is above the next entry).
            const float ev = (job_ok && !fb) ? eps : 0.0f;
            int walked_b = 0;
            if (LOW && b_form == 2) {
                // no Z: every sample counts in n_z, and n_xz is a range of the
                // job's sorted X column (a permutation does not change it)
                nz = ev > 0.0f ? static_cast<int>(a.n) - 1 : 0;
                nxz = count_sorted(a.xsort + static_cast<int64_t>(a.jobs[job_ok ? job : 0].x) * a.n,
                                   static_cast<int>(a.n), xq[0], ev);
            }
            // b_form 1: one z column, and the order is by it: the samples on
            // either side of the query take the place of the list
            const int parts_b = !LOW || b_form == 0 ? 1 : (b_form == 1 ? 2 : 0);
#pragma unroll 1
            for (int part = 0; part < parts_b; ++part) {
                const Src lb = LOW && b_form == 1
                                   ? side(part ? -1 : 1, 0)
                                   : Src{a.list_b + static_cast<int64_t>(qi) * a.cap_b, __ldg(&a.lmeta[qi].y), 0, 0};
                int pos = 0;
                uint32_t rem;
                begin(lb);
                while (true) {
                    rem = __ballot_sync(kFull, ev > row_d[0]);
                    if (__popc(rem) <= IDTX_LIST_REPACK) break;
                    float dx[SW], dz[SW];
#pragma unroll
                    for (int t = 0; t < SW; ++t) {
                        dx[t] = fabsf(xq[0] - row_x[t][0]);
#pragma unroll
                        for (int d = 1; d < DX; ++d) dx[t] = fmaxf(dx[t], fabsf(xq[d] - row_x[t][d]));
                        dz[t] = row_d[t];
                    }
                    advance(lb, pos);
                    pos += SW;
#pragma unroll
                    for (int t = 0; t < SW; ++t) {
                        const bool pz = dz[t] < ev;
                        if (!SEARCH_Z) nz += pz ? 1 : 0;
                        nxz += (pz && dx[t] < ev) ? 1 : 0;
                    }
                }
                walked_b += pos < lb.len ? pos : lb.len;
                // The jobs that need more share the lanes: with c of them left,
                // M slots (the power of two >= c) of 32 / M lanes that split the
                // entries between them; once at most M / 2 need more, the lanes
                // are shared out again.
                while (rem) {
                    const int c = __popc(rem);
                    const int lg = c > 8 ? 4 : (c > 4 ? 3 : (c > 2 ? 2 : (c > 1 ? 1 : 0)));
                    const int M = 1 << lg, per = 32 >> lg;
                    const int s = lane & (M - 1), r = lane >> lg;
                    const int rank = __popc(rem & ((1u << lane) - 1u));
                    int *tab = &ent[0].x;  // the staged entries are done with
                    __syncwarp();
                    if ((rem >> lane) & 1u) tab[rank] = lane;
                    __syncwarp();
                    const int home = s < c ? tab[s] : lane;
                    const float e_home = __shfl_sync(kFull, ev, home);
                    const float es = s < c ? e_home : 0.0f;
                    float xs[DX];
#pragma unroll
                    for (int d = 0; d < DX; ++d) xs[d] = __shfl_sync(kFull, xq[d], home);
                    const float *xgs = xg + (home - lane) * DX;
                    const int from = pos;
                    int cz = 0, cx = 0;
                    uint32_t still;
                    do {
                        constexpr int PS = DX == 1 ? IDTX_LIST_PHASE_STEP : 4;
                        int js[PS];
                        float xv[PS][DX];
#pragma unroll
                        for (int t = 0; t < PS; ++t) {
                            const int e = pos + r + per * t;
                            const int2 v = entry(lb, e);
                            js[t] = __int_as_float(v.y) < es ? v.x : -1;
                        }
#pragma unroll
                        for (int t = 0; t < PS; ++t) {
#pragma unroll
                            for (int d = 0; d < DX; ++d) xv[t][d] = CUDART_INF_F;
                            if (js[t] >= 0)
                                load_x<DX>(xgs + static_cast<uint64_t>(static_cast<uint32_t>(js[t])) * XW, xv[t]);
                        }
                        pos += per * PS;
                        const float dn = pos < lb.len ? entry_d(lb, pos) : kInf;
#pragma unroll
                        for (int t = 0; t < PS; ++t) {
                            float dxv = fabsf(xs[0] - xv[t][0]);
#pragma unroll
                            for (int d = 1; d < DX; ++d) dxv = fmaxf(dxv, fabsf(xs[d] - xv[t][d]));
                            if (!SEARCH_Z) cz += js[t] >= 0 ? 1 : 0;
                            cx += dxv < es ? 1 : 0;
                        }
                        still = __ballot_sync(kFull, ((rem >> lane) & 1u) && ev > dn);
                    } while (__popc(still) > (M >> 1));
                    tb += static_cast<unsigned>(c * (pos - from));
                    // each slot's totals over its lanes, then to the job's lane
                    for (int off = M; off < 32; off <<= 1) {
                        if (!SEARCH_Z) cz += __shfl_xor_sync(kFull, cz, off);
                        cx += __shfl_xor_sync(kFull, cx, off);
                    }
                    const int vz = SEARCH_Z ? 0 : __shfl_sync(kFull, cz, rank & 31);
                    const int vx = __shfl_sync(kFull, cx, rank & 31);
                    if ((rem >> lane) & 1u) {
                        nz += vz;
                        nxz += vx;
                    }
                    rem = still;
                }
                if (SEARCH_Z) {  // n_z, of the entries that the walk reached
                    const int hi = pos < lb.len ? pos : lb.len;
                    int lo = 0;
                    for (int b = 1 << (31 - __clz(hi | 1)); b; b >>= 1)
                        if (lo + b <= hi && entry_d(lb, lo + b - 1) < ev) lo += b;
                    nz += lo;
                }
            }
            // Jobs whose eps reaches past a list are left to ksg_scan_kernel.
            const uint32_t bmask = __ballot_sync(kFull, fb);
            nfb = __popc(bmask);
            if (bmask) {
                // the jobs, and those of them whose eps is not known yet
                const uint32_t amask = __ballot_sync(kFull, fa);
                if (lane == 0) {
                    const bool few = __popc(bmask) <= kFewJobs;
                    const int64_t i = atomicAdd(a.next + (few ? 2 : 3), 1);
                    a.scans[few ? i : static_cast<int64_t>(n_groups) * a.n_pad - 1 - i] =
                        make_int4(grp, qi, static_cast<int>(bmask), static_cast<int>(amask));
                }
                // eps, or a bound of it, in the place of the counts to come
                if (fb) {
                    nz = __float_as_int(eps);
                    nyz = static_cast<int>(__float_as_uint(eps) >> 16);
                }
            }
            const int64_t at = (static_cast<int64_t>(grp) * a.n_pad + qi) * GB + lane;
            put_count(a.cyz, at, nyz, a.wide);
            put_count(a.cz, at, nz, a.wide);
            put_count(a.cxz, at, nxz, a.wide);
            if (a.eps_out && job_ok && !fb) {
                const int64_t orig = a.order ? static_cast<int64_t>(a.order[qi]) : static_cast<int64_t>(qi);
                a.eps_out[static_cast<int64_t>(job) * a.n + orig] = eps;
            }
            if (a.work) {
                // lane k keeps counter k: no read-modify-write per query
                // (sum_terms has the sums of n_z and n_yz)
                unsigned v = static_cast<unsigned>(walked_a);
                v = lane == 1 ? static_cast<unsigned>(walked_b) : v;
                v = lane == 6 ? tb : v;
                v = lane == 7 ? ta : v;
                my_work += lane < 2 || lane == 6 || lane == 7 ? v : 0u;
                if (nfa | nfb) {
                    const unsigned long long n1 = static_cast<unsigned long long>(a.n - 1);
                    my_work += lane == 2 ? nfa * n1 : (lane == 3 ? nfb * n1 : (lane == 4 ? nfa + nfb : 0ull));
                }
            }
        }
    }

    if (lane == 5) my_work = static_cast<unsigned long long>(clock64() - t_begin);
    if (lane < kNumWork) sm.work[warp][lane] = my_work;
    __syncthreads();
    if (tid == 0) {  // the last CTA to come here resets the counters for the next launch
        __threadfence();
        if (atomicAdd(a.next + 1, 1) == static_cast<int>(gridDim.x) - 1) {
            a.next[0] = 0;
            a.next[1] = 0;
        }
    }
    if (a.work && tid < kNumWork) {
        unsigned long long s = 0;
        for (int w = 0; w < NW; ++w) s += sm.work[w][tid];
        atomicAdd(&a.work[tid], s);
    }
}

// Full scans, for the (query, group)s that the lists did not serve: the counts
// of the marked jobs over every sample, and first eps where it is not known yet
// (item.w).  A query far from the others has long
// neighbourhoods for all of its jobs; far more often one or two jobs of a query
// have an outlying x, so that their neighbourhoods reach past the lists: of
// 1611 items at N = 9995, three z, lists of 512 and 1024, 96 surrogates, 1311
// had one job and 56 more than eight.  So there are two ways:
//   * More than kFewJobs jobs: a CTA takes one item at a time, each of its warps
//     32 samples of every eighth tile; in a warp a lane per sample finds the
//     samples within reach, 32 at a time, and a lane per job uses them, their X
//     rows loaded sixteen at a time.  (A single warp of the list kernel took up
//     to 1 ms for one such query at N = 9995 with 32 jobs; 70 us here.)
//   * Fewer: the CTA's four quarters take one item each, a lane per sample; the
//     jobs' x values are loaded where the subspace distance is within reach, of
//     four segments of 32 samples at once, and the counts are votes.
// The warps share each job's smallest k-th distance so far (any warp's is at
// least the job's own) and their heaps and counts meet in shared memory.
// Both are bound by the latency of their loads.  Measured, N = 9995, 101
// estimates, against the first way for every item with eps sought afresh: two
// z columns, lists of 512 and 1024 (10117 scanned jobs), 978 -> 147 us; three
// z, 556 -> 98 us; 2001 estimates (99543), 9.4 -> 1.4 ms.  Scans are then so
// much cheaper that shorter lists win: the first call 1.43 -> 0.98 ms.
constexpr int kScanWarps = 32;
constexpr int kScanQuarter = kScanWarps / 4;
static_assert(kScanQuarter % (kTJ / 32) == 0, "whole tiles per step");

template <int DX, int DY, int DZ, int K1, bool EXACT, int QCTA, int NWARPS>
__global__ void __launch_bounds__(kScanWarps * 32, 1)
    ksg_scan_kernel(const KsgLaunch a)
{
    using S = KsgShape<DX, DY, DZ, K1, EXACT, QCTA, NWARPS>;
    constexpr int DS = S::DS, DSP = S::DSP, XW = S::XW, GB = S::GB;
    constexpr int KH = K1 - 1, U = DX > 1 ? 8 : 16;
    constexpr unsigned kFull = 0xffffffffu;
    extern __shared__ __align__(16) unsigned char l_smem[];
    float(*s_heap)[KH][32] = reinterpret_cast<float(*)[KH][32]>(l_smem);  // [kScanWarps]
    __shared__ unsigned s_th[32];  // bits of each job's bound, then of its eps
    __shared__ int s_cnt[3][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int n = static_cast<int>(a.n), n_tiles = (n + kTJ - 1) / kTJ;
    const int n_few = a.next[2], n_many = a.next[3], kk = a.k;
    const int4 *many = a.scans + static_cast<int64_t>((a.n_jobs + GB - 1) / GB) * a.n_pad - 1;
    auto kth = [&](const float(&h)[KH]) { return EXACT ? h[KH - 1] : select_kth<KH>(h, kk - 1); };
    // eps of a job, or a bound of it, as the list kernel left it
    auto left = [&](int64_t at) {
        const unsigned v = static_cast<unsigned>(get_count(a.cz, at, a.wide));
        return a.wide ? v : v | static_cast<unsigned>(get_count(a.cyz, at, 0)) << 16;
    };
    for (int it = blockIdx.x; it < n_many; it += gridDim.x) {
        const int4 item = many[-it];
        const int grp = item.x, qi = item.y;
        const bool mine = (static_cast<unsigned>(item.z) >> lane) & 1u;  // this lane's job is wanted
        const bool seek = (static_cast<unsigned>(item.w) >> lane) & 1u;  // and its eps
        const int64_t at = (static_cast<int64_t>(grp) * a.n_pad + qi) * GB + lane;
        const float *xg = a.xi + static_cast<int64_t>(grp) * a.n_pad * XW + lane * DX;
        float xq[DX], q[DS];
        load_x<DX>(xg + static_cast<int64_t>(qi) * XW, xq);
        const float *qr = a.sh + (static_cast<int64_t>(qi / kTJ) * kTileRows + qi % kTJ) * DSP;
#pragma unroll
        for (int d = 0; d < DS; ++d) q[d] = qr[d];
        // use(d_X, d_Z, d_YZ of U samples) for every sample j != qi of the
        // warp's tiles with d_YZ (ZONLY: d_Z) below limit() as it was before
        // its 32 samples
        auto scan = [&](auto zonly, auto limit, auto use) {
            constexpr bool ZONLY = decltype(zonly)::value;
            constexpr int SEGS = kTJ / 32, STEP = kScanWarps / SEGS;  // a warp: one segment of every STEP-th tile
            const int b = warp % SEGS * 32;
            float lim = limit();
            for (int i0 = 0; i0 * STEP < n_tiles; i0 += 32) {
                // from the query's own tile outwards, so that the bounds are
                // soon tight; 32 tiles' boxes are tested at a time
                const int u = (i0 + lane) * STEP + warp / SEGS;
                const int my_tile = u < n_tiles ? spiral_tile(qi / kTJ, n_tiles, u) : 0;
                const float my_gap =
                    u < n_tiles ? point_gap<ZONLY ? DZ : DS, DSP>(
                                      a.sh + static_cast<int64_t>(my_tile) * kTileRows * DSP, q)
                                : CUDART_INF_F;
                uint32_t todo = __ballot_sync(kFull, my_gap < lim);
                while (todo) {
                    const int w = __ffs(todo) - 1;
                    todo &= todo - 1;
                    const int t = __shfl_sync(kFull, my_tile, w);
                    if (!(__shfl_sync(kFull, my_gap, w) < lim)) continue;
                    const float *row = a.sh + (static_cast<int64_t>(t) * kTileRows + b + lane) * DSP;
                    float dz = fabsf(q[0] - row[0]);
#pragma unroll
                    for (int d = 1; d < DZ; ++d) dz = fmaxf(dz, fabsf(q[d] - row[d]));
                    float dyz = dz;
#pragma unroll
                    for (int d = DZ; d < DS; ++d) dyz = fmaxf(dyz, fabsf(q[d] - row[d]));
                    const int j0 = t * kTJ + b;
                    const bool other = j0 + lane < n && j0 + lane != qi;
                    uint32_t in = __ballot_sync(kFull, other && (ZONLY ? dz : dyz) < lim);
                    while (in) {
                        float dx[U], z[U], yz[U];  // +inf where no sample is left
#pragma unroll
                        for (int v = 0; v < U; ++v) {
                            const int s = __ffs(in) - 1;
                            const bool some = in != 0;
                            in &= in - 1;
                            float xr[DX];
                            load_x<DX>(xg + static_cast<int64_t>(some ? j0 + s : qi) * XW, xr);
                            dx[v] = fabsf(xq[0] - xr[0]);
#pragma unroll
                            for (int d = 1; d < DX; ++d) dx[v] = fmaxf(dx[v], fabsf(xq[d] - xr[d]));
                            z[v] = __shfl_sync(kFull, dz, s & 31);
                            yz[v] = __shfl_sync(kFull, dyz, s & 31);
                            if (!some) z[v] = yz[v] = CUDART_INF_F;
                        }
                        use(dx, z, yz);
                    }
                    lim = limit();
                }
            }
        };
        if (warp == 0) {
            s_th[lane] = mine ? left(at) : 0u;
            s_cnt[0][lane] = s_cnt[1][lane] = s_cnt[2][lane] = 0;
        }
        __syncthreads();
        volatile unsigned *th_all = s_th;
        float h[KH];
#pragma unroll
        for (int t = 0; t < KH; ++t) h[t] = CUDART_INF_F;
        float th = seek ? CUDART_INF_F : 0.0f;  // other jobs do not raise the limit
        // A distance equal to the shared bound may be the k-th itself, so the
        // limit is the next float above it.
        if (item.w) scan(std::false_type{},
             [&] {
                 if (seek && th < __uint_as_float(th_all[lane])) atomicMin(&s_th[lane], __float_as_uint(th));
                 const unsigned m = __reduce_max_sync(kFull, min(th_all[lane], __float_as_uint(th)));
                 return m < 0x7f800000u ? __uint_as_float(m + 1) : CUDART_INF_F;
             },
             [&](const float(&dx)[U], const float(&)[U], const float(&yz)[U]) {
                 if constexpr (EXACT && KH == 4) {
#pragma unroll
                     for (int u = 0; u < U; u += 4)
                         merge4(h, fmaxf(dx[u], yz[u]), fmaxf(dx[u + 1], yz[u + 1]),
                                fmaxf(dx[u + 2], yz[u + 2]), fmaxf(dx[u + 3], yz[u + 3]));
                 } else {
#pragma unroll
                     for (int u = 0; u < U; ++u) {
                         const float d = fmaxf(dx[u], yz[u]);
                         if (d < kth(h)) sorted_insert<KH>(h, d);
                     }
                 }
                 if (seek) th = kth(h);
             });
        if (item.w) {
#pragma unroll
            for (int t = 0; t < KH; ++t) s_heap[warp][t][lane] = h[t];
            __syncthreads();
            if (warp == 0) {  // the k smallest of all warps
                for (int w = 1; w < kScanWarps; ++w)
                    for (int t = 0; t < KH; ++t) {
                        const float d = s_heap[w][t][lane];
                        if (!__any_sync(kFull, seek && d < kth(h))) break;
                        if (d < kth(h)) sorted_insert<KH>(h, d);
                    }
                if (seek) s_th[lane] = __float_as_uint(kth(h));
            }
            __syncthreads();
        }
        const float eps = __uint_as_float(s_th[lane]);
        const float lim = warp_max_nn(eps);
        int cz = 0, cyz = 0, cxz = 0;
        scan(std::true_type{}, [&] { return lim; },
             [&](const float(&dx)[U], const float(&z)[U], const float(&yz)[U]) {
#pragma unroll
                 for (int u = 0; u < U; ++u) {
                     cz += z[u] < eps ? 1 : 0;
                     cyz += yz[u] < eps ? 1 : 0;
                     cxz += (z[u] < eps && dx[u] < eps) ? 1 : 0;
                 }
             });
        if (cz) {
            atomicAdd(&s_cnt[0][lane], cz);
            if (cyz) atomicAdd(&s_cnt[1][lane], cyz);
            if (cxz) atomicAdd(&s_cnt[2][lane], cxz);
        }
        __syncthreads();
        if (warp == 0 && mine) {
            put_count(a.cz, at, s_cnt[0][lane], a.wide);
            put_count(a.cyz, at, s_cnt[1][lane], a.wide);
            put_count(a.cxz, at, s_cnt[2][lane], a.wide);
            if (a.eps_out) {
                const int64_t orig = a.order ? static_cast<int64_t>(a.order[qi]) : static_cast<int64_t>(qi);
                a.eps_out[static_cast<int64_t>(grp * GB + lane) * a.n + orig] = eps;
            }
        }
        __syncthreads();  // shared state is set up afresh by the next item
    }

    // ---------------- items of few jobs, by quarters of the CTA
    constexpr int V = DSP <= 4 ? 4 : (DSP <= 12 ? 2 : 1);  // segments of 32 samples at once
    __shared__ unsigned s_bound[4][kFewJobs];  // bits of each job's bound, then of its eps
    __shared__ int s_few[4][3][kFewJobs], s_item[4];
    const int part = warp / kScanQuarter, pw = warp % kScanQuarter;
    auto part_sync = [&] {
        asm volatile("bar.sync %0, %1;" ::"r"(1 + part), "n"(kScanQuarter * 32) : "memory");
    };
    while (true) {
        if (pw == 0 && lane == 0) s_item[part] = atomicAdd(a.next + 4, 1);
        part_sync();
        const int it = s_item[part];
        if (it >= n_few) break;
        const int4 item = a.scans[it];
        const int grp = item.x, qi = item.y, m = __popc(item.z);
        // lane l < m serves the l-th marked job
        uint32_t rest = static_cast<uint32_t>(item.z);
        for (int t = 0; t < lane && t + 1 < m; ++t) rest &= rest - 1;
        const int job = __ffs(rest) - 1;
        const bool mine = lane < m, seek = mine && ((static_cast<uint32_t>(item.w) >> job) & 1u);
        const uint32_t seeks = __ballot_sync(kFull, seek);
        const int64_t at = (static_cast<int64_t>(grp) * a.n_pad + qi) * GB + job;
        const float *xg = a.xi + static_cast<int64_t>(grp) * a.n_pad * XW;
        float xq[DX], q[DS];
        load_x<DX>(xg + static_cast<int64_t>(qi) * XW + job * DX, xq);
        const float *qr = a.sh + (static_cast<int64_t>(qi / kTJ) * kTileRows + qi % kTJ) * DSP;
#pragma unroll
        for (int d = 0; d < DS; ++d) q[d] = qr[d];
        if (pw == 0 && mine) {
            s_bound[part][lane] = left(at);
            s_few[part][0][lane] = s_few[part][1][lane] = s_few[part][2][lane] = 0;
        }
        part_sync();
        volatile unsigned *bound = s_bound[part];
        // use(samples, d_Z, d_YZ) of V samples a lane (+inf: none), for the tiles
        // whose d_YZ (ZONLY: d_Z) may be below limit()
        auto sweep = [&](auto zonly, auto limit, auto use) {
            constexpr bool ZONLY = decltype(zonly)::value;
            constexpr int SEGS = kTJ / 32, STEP = kScanQuarter / SEGS;
            const int b = pw % SEGS * 32;
            float lim = limit();
            for (int i0 = 0; i0 * STEP < n_tiles; i0 += 32) {
                const int u = (i0 + lane) * STEP + pw / SEGS;
                const int my_tile = u < n_tiles ? spiral_tile(qi / kTJ, n_tiles, u) : 0;
                const float my_gap =
                    u < n_tiles ? point_gap<ZONLY ? DZ : DS, DSP>(
                                      a.sh + static_cast<int64_t>(my_tile) * kTileRows * DSP, q)
                                : CUDART_INF_F;
                uint32_t todo = __ballot_sync(kFull, my_gap < lim);
                while (todo) {
                    int j[V];
                    float dz[V], dyz[V];
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        const int t = todo ? __shfl_sync(kFull, my_tile, (__ffs(todo) - 1) & 31) : -1;
                        todo &= todo - 1;
                        j[v] = t * kTJ + b + lane;
                        const bool some = t >= 0 && j[v] < n && j[v] != qi;
                        if (!some) j[v] = qi;
                        const float4 *row = reinterpret_cast<const float4 *>(
                            t >= 0 ? a.sh + (static_cast<int64_t>(t) * kTileRows + b + lane) * DSP : qr);
                        float r[DSP];
#pragma unroll
                        for (int c = 0; c < DSP / 4; ++c) {
                            const float4 f = row[c];
                            r[4 * c] = f.x;
                            r[4 * c + 1] = f.y;
                            r[4 * c + 2] = f.z;
                            r[4 * c + 3] = f.w;
                        }
                        dz[v] = some ? fabsf(q[0] - r[0]) : CUDART_INF_F;
#pragma unroll
                        for (int d = 1; d < DZ; ++d) dz[v] = fmaxf(dz[v], fabsf(q[d] - r[d]));
                        dyz[v] = dz[v];
#pragma unroll
                        for (int d = DZ; d < DS; ++d) dyz[v] = fmaxf(dyz[v], fabsf(q[d] - r[d]));
                    }
                    use(j, dz, dyz);
                    lim = limit();
                    todo &= __ballot_sync(kFull, my_gap < lim);
                }
            }
        };
        // d_X of the l-th job to V samples, +inf where `near` is false
        auto x_dists = [&](int l, const int(&j)[V], const bool(&near)[V], float(&dx)[V]) {
            const float *xj = xg + __shfl_sync(kFull, job, l) * DX;
            float xl[DX];
#pragma unroll
            for (int d = 0; d < DX; ++d) xl[d] = __shfl_sync(kFull, xq[d], l);
#pragma unroll
            for (int v = 0; v < V; ++v) {
                float xr[DX];
#pragma unroll
                for (int d = 0; d < DX; ++d) xr[d] = CUDART_INF_F;
                if (near[v]) load_x<DX>(xj + static_cast<int64_t>(j[v]) * XW, xr);
                dx[v] = fabsf(xl[0] - xr[0]);
#pragma unroll
                for (int d = 1; d < DX; ++d) dx[v] = fmaxf(dx[v], fabsf(xl[d] - xr[d]));
            }
        };
        // the next float above a bound: a distance equal to it may be the k-th
        auto above = [](unsigned bits) {
            return __uint_as_float(bits < 0x7f800000u ? bits + 1 : 0x7f800000u);
        };
        if (seeks) {
            float h[KH];  // lane l: the l-th job's smallest distances
#pragma unroll
            for (int t = 0; t < KH; ++t) h[t] = CUDART_INF_F;
            sweep(std::false_type{},
                  [&] { return above(__reduce_max_sync(kFull, seek ? bound[lane] : 0u)); },
                  [&](const int(&j)[V], const float(&)[V], const float(&dyz)[V]) {
                      for (uint32_t left_l = seeks; left_l; left_l &= left_l - 1) {
                          const int l = __ffs(left_l) - 1;
                          const unsigned was = __shfl_sync(kFull, bound[l], 0);
                          const float lim = above(was);
                          bool near[V];
#pragma unroll
                          for (int v = 0; v < V; ++v) near[v] = dyz[v] < lim;
                          float dx[V];
                          x_dists(l, j, near, dx);
#pragma unroll
                          for (int v = 0; v < V; ++v) {
                              const float d = fmaxf(dx[v], dyz[v]);
                              uint32_t hits = __ballot_sync(kFull, d < lim);
                              while (hits) {
                                  const float dh = __shfl_sync(kFull, d, __ffs(hits) - 1);
                                  hits &= hits - 1;
                                  if (lane == l && dh < kth(h)) sorted_insert<KH>(h, dh);
                              }
                          }
                          if (lane == l && __float_as_uint(kth(h)) < was)
                              atomicMin(&s_bound[part][l], __float_as_uint(kth(h)));
                      }
                  });
#pragma unroll
            for (int t = 0; t < KH; ++t) s_heap[warp][t][lane] = h[t];
            part_sync();
            if (pw == 0 && seek) {  // the k smallest of the quarter's warps
                for (int w = 1; w < kScanQuarter; ++w)
                    for (int t = 0; t < KH; ++t) {
                        const float d = s_heap[warp + w][t][lane];
                        if (!(d < kth(h))) break;
                        sorted_insert<KH>(h, d);
                    }
                s_bound[part][lane] = __float_as_uint(kth(h));
            }
            part_sync();
        }
        const float eps = mine ? __uint_as_float(bound[lane]) : 0.0f;
        const float lim = warp_max_nn(eps);
        int cz = 0, cyz = 0, cxz = 0;
        sweep(std::true_type{}, [&] { return lim; },
              [&](const int(&j)[V], const float(&dz)[V], const float(&dyz)[V]) {
                  for (int l = 0; l < m; ++l) {
                      const float el = __shfl_sync(kFull, eps, l);
                      bool near[V];
#pragma unroll
                      for (int v = 0; v < V; ++v) near[v] = dz[v] < el;
                      float dx[V];
                      x_dists(l, j, near, dx);
                      int c0 = 0, c1 = 0, c2 = 0;
#pragma unroll
                      for (int v = 0; v < V; ++v) {
                          c0 += __popc(__ballot_sync(kFull, near[v]));
                          c1 += __popc(__ballot_sync(kFull, dyz[v] < el));
                          c2 += __popc(__ballot_sync(kFull, dx[v] < el));
                      }
                      if (lane == l) {
                          cz += c0;
                          cyz += c1;
                          cxz += c2;
                      }
                  }
              });
        if (mine) {
            atomicAdd(&s_few[part][0][lane], cz);
            atomicAdd(&s_few[part][1][lane], cyz);
            atomicAdd(&s_few[part][2][lane], cxz);
        }
        part_sync();
        if (pw == 0 && mine) {
            put_count(a.cz, at, s_few[part][0][lane], a.wide);
            put_count(a.cyz, at, s_few[part][1][lane], a.wide);
            put_count(a.cxz, at, s_few[part][2][lane], a.wide);
            if (a.eps_out) {
                const int64_t orig = a.order ? static_cast<int64_t>(a.order[qi]) : static_cast<int64_t>(qi);
                a.eps_out[static_cast<int64_t>(grp * GB + job) * a.n + orig] = eps;
            }
        }
    }
    // the last CTA to come here empties the queue for the next launch
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(a.next + 1, 1) == static_cast<int>(gridDim.x) - 1) {
            for (int t = 1; t < 5; ++t) a.next[t] = 0;
        }
    }
}

// The estimates of n_groups groups, as many at a time as the count buffers
// hold: the list kernel, the scans it left, the sums.  n_qt * n_groups <= 0
// only sets up.
template <int DX, int DY, int DZ, int K1, bool EXACT, int QC, int NWARPS>
cudaError_t launch_ksg_list(const KsgLaunch &all, int n_groups, cudaStream_t stream)
{
    using LS = ListShape<DX, DY, DZ, K1, EXACT, QC, NWARPS>;
    using S = typename LS::S;
    auto kern = ksg_list_kernel<DX, DY, DZ, K1, EXACT, QC, NWARPS>;
    auto scan = ksg_scan_kernel<DX, DY, DZ, K1, EXACT, QC, NWARPS>;
    constexpr size_t kScanSmem = kScanWarps * (K1 - 1) * 32 * sizeof(float);
    // Per device: the dynamic shared memory, a carveout that leaves the rest
    // of the SM's memory to L1, and the SM count (one CTA per SM).
    static DeviceOnce setup;
    static int n_sms[kMaxDevices];
    cudaError_t e = once_per_device(setup, [&](int d) {
        cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(LS::SMEM));
        if (r == cudaSuccess) {
            int smem_sm = 0;
            r = cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, d);
            if (r == cudaSuccess && smem_sm > 0) {
                const int pct = static_cast<int>((LS::SMEM + 1024) * 100 / smem_sm) + 1;
                r = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout,
                                         pct < 100 ? pct : 100);
            }
        }
        if (r == cudaSuccess) r = cudaDeviceGetAttribute(&n_sms[d], cudaDevAttrMultiProcessorCount, d);
        if (r == cudaSuccess)
            r = cudaFuncSetAttribute(scan, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     static_cast<int>(kScanSmem));
        return r;
    });
    if (e != cudaSuccess || static_cast<int64_t>(all.n_qt) * n_groups <= 0) return e;
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (all.count_groups < 1) return cudaErrorInvalidValue;
    for (int g0 = 0; g0 < n_groups; g0 += all.count_groups) {
        const int groups = n_groups - g0 < all.count_groups ? n_groups - g0 : all.count_groups;
        const int64_t j0 = static_cast<int64_t>(g0) * S::GB;
        KsgLaunch a = all;
        a.n_jobs = static_cast<int>(all.n_jobs - j0 < groups * S::GB ? all.n_jobs - j0 : groups * S::GB);
        a.xi += g0 * all.n_pad * S::XW;
        a.partial += j0 * all.n_qt;
        if (a.eps_out) a.eps_out += j0 * all.n;
        if (a.cnt_out) a.cnt_out += j0 * 3 * all.n;
        if (a.jobs) a.jobs += j0;
        // Chunks of consecutive queries: eight per SM where that leaves 16 queries,
        // else 16, or, if these would leave SMs without any, one per SM of at
        // least four (the queries of a small call are one wave of warps: 21
        // estimates, one z column, dx = 3, N = 1000, 192 us in chunks of 16, 93 in 143
        // of 7; k = 4, two z columns, 23.8 and 20.9; one estimate, N = 129, 8.2 in
        // chunks of 16, 7.4 of four, 12.9 of one, most of a CTA's warps in each
        // other's way to it).
        const int64_t per = a.n * groups / (8 * n_sms[dev]);
        const int64_t one = (a.n * groups + n_sms[dev] - 1) / n_sms[dev];
        const int64_t few = one < 4 ? 4 : (one < 16 ? one : 16);
        const int chunk = static_cast<int>(per > IDTX_LIST_CHUNKQ ? IDTX_LIST_CHUNKQ : (per >= 16 ? per : few));
        const int64_t chunks = groups * ((a.n + chunk - 1) / chunk);
        if (chunks > 0x3fffffff) return cudaErrorInvalidValue;  // the kernel's chunk arithmetic is 32-bit
        const int64_t grid = chunks < n_sms[dev] ? chunks : n_sms[dev];
        kern<<<static_cast<unsigned>(grid), LS::THREADS, LS::SMEM, stream>>>(
            a, groups, static_cast<int>(chunks), chunk);
        scan<<<static_cast<unsigned>(n_sms[dev]), kScanWarps * 32, kScanSmem, stream>>>(a);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = sum_terms(a, QC, groups, n_sms[dev], stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// One compiled specialisation: the tile kernel (ksg_kernel.cuh), its
// persistent form, the list kernel with the same query tiles, and the plain
// schedule (ksg_plain.cuh) of the same dimension bucket.
template <int DX, int DY, int DZ, int K1, bool EXACT, int QC, int NWARPS>
KsgVariant make_variant()
{
    using S = KsgShape<DX, DY, DZ, K1, EXACT, QC, NWARPS>;
    return KsgVariant{DX, DY, DZ, K1, EXACT ? 1 : 0, S::GB, S::DSP, S::QC,
                      &launch_ksg<DX, DY, DZ, K1, EXACT, QC, NWARPS>,
                      &launch_ksg_table<DX, DY, DZ, K1, EXACT, QC, NWARPS>,
                      &launch_ksg_list<DX, DY, DZ, K1, EXACT, QC, NWARPS>,
                      &launch_ksg_plain<DX, DY, DZ, K1, EXACT, QC, NWARPS>};
}

}  // namespace idtx
