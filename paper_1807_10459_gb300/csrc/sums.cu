// sums.cu -- the digamma terms of the list kernel's counts and their sums.
#include <cuda_runtime.h>

#include "ksg_common.cuh"

namespace idtx {

namespace {

// Tiles of qc queries of one group, in turn.  A lane takes four jobs of a query
// (8 lanes a query, four queries a warp), so its counts come in 8-byte loads,
// two queries' in flight; the lanes' and warps' sums are added at the end.
// Bound by the table lookups (the counts are 6 bytes a query and job), so with
// many tiles a block first takes the table's first kTable entries into shared
// memory, which nearly all counts are below (a gather there costs its bank
// conflicts, three to four, and in L1 a cycle for every line).
// N = 9995, 9447 estimates: 0.58 -> 0.30 ms against terms and sums in fp64, of
// which an SM does two operations a clock (see kPsiBits), 0.27 with the
// table in shared memory; N = 4997, 28 thousand: 0.89 -> 0.51 -> 0.38.
constexpr int kRowsPerWarp = 8, kTable = 2048;
template <typename Four, bool TABLE>  // four counts: uint2 of 16 bits each, uint4 of 32
__global__ void k_sum_terms(const KsgLaunch a, int qc, int64_t n_tasks)
{
    extern __shared__ __align__(16) long long s_psi[];  // TABLE: [kTable]
    __shared__ long long s_sum[8][32];  // [warp][job]
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int j0 = (lane & 7) * 4;
    unsigned long long sz = 0, syz = 0;  // for the work counters
    if (TABLE) {
        const int top = (int)min((int64_t)kTable, a.n + 1);
        for (int t = threadIdx.x; t < top; t += blockDim.x) s_psi[t] = __ldg(a.psi + t);
        __syncthreads();
    }
    auto psi = [&](int c) { return TABLE && c < kTable ? s_psi[c] : __ldg(a.psi + c); };
    for (int64_t task = blockIdx.x; task < n_tasks; task += gridDim.x) {
        const int grp = (int)(task / a.n_qt), qt = (int)(task - (int64_t)grp * a.n_qt);
        const int n_job = min(4, a.n_jobs - (grp * 32 + j0));
        const int64_t q0 = (int64_t)qt * qc;
        long long sum[4] = {0, 0, 0, 0};
        constexpr int kRows = kRowsPerWarp / 4;
        Four z[kRows], xz[kRows], yz[kRows];
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            const int64_t qi = min(q0 + w * kRowsPerWarp + u * 4 + (lane >> 3), a.n_pad - 1);
            const int64_t at = (((int64_t)grp * a.n_pad + qi) * 32 + j0) / 4;
            z[u] = __ldcs(static_cast<const Four *>(a.cz) + at);
            xz[u] = __ldcs(static_cast<const Four *>(a.cxz) + at);
            yz[u] = __ldcs(static_cast<const Four *>(a.cyz) + at);
        }
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            const int m = w * kRowsPerWarp + u * 4 + (lane >> 3);
            const int64_t qi = q0 + m;
            if (m >= qc || qi >= a.n) continue;
            const int64_t orig = a.cnt_out && a.order ? (int64_t)a.order[qi] : qi;
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                if (t >= n_job) break;
                auto part = [&](const Four &v) {
                    if constexpr (sizeof(Four) == sizeof(uint4)) {
                        // within psi's table also where the list kernel gave up
                        const unsigned c = t == 0 ? v.x : (t == 1 ? v.y : (t == 2 ? v.z : v.w));
                        return (int)min(c, (unsigned)a.n - 1u);
                    } else {  // (the table has at least 65536 entries)
                        return (int)((t < 2 ? v.x : v.y) >> (t & 1) * 16 & 0xffffu);
                    }
                };
                const int nz = part(z[u]), nxz = part(xz[u]), nyz = part(yz[u]);
                sz += nz;
                syz += nyz;
                sum[t] += psi(nz + 1) - psi(nxz + 1) - psi(nyz + 1);
                if (a.cnt_out) {
                    int32_t *co = a.cnt_out + (int64_t)(grp * 32 + j0 + t) * 3 * a.n;
                    co[orig] = nxz;
                    co[a.n + orig] = nyz;
                    co[2 * a.n + orig] = nz;
                }
            }
        }
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            sum[t] += __shfl_xor_sync(0xffffffffu, sum[t], 8);
            sum[t] += __shfl_xor_sync(0xffffffffu, sum[t], 16);
            if (lane < 8) s_sum[w][j0 + t] = sum[t];
        }
        __syncthreads();
        const int job = grp * 32 + lane;
        if (w == 0 && job < a.n_jobs) {
            long long s = 0;
            for (int v = 0; v < nw; ++v) s += s_sum[v][lane];
            a.partial[(int64_t)job * a.n_qt + qt] = s;
        }
        __syncthreads();
    }
    if (a.work) {
        for (int o = 16; o >= 1; o >>= 1) {
            sz += __shfl_xor_sync(0xffffffffu, sz, o);
            syz += __shfl_xor_sync(0xffffffffu, syz, o);
        }
        if (lane < 2) atomicAdd(&a.work[8 + lane], lane ? syz : sz);
    }
}

template <typename Four>
cudaError_t launch_sum(const KsgLaunch &a, int qc, int64_t n_tasks, int n_sms, cudaStream_t st)
{
    // With the table: as many blocks as the SMs hold, when each then has at
    // least four tiles to take.
    const int64_t blocks = n_sms * 8;
    const unsigned threads = (unsigned)(qc / kRowsPerWarp * 32);
    if (n_tasks >= 4 * blocks)
        k_sum_terms<Four, true><<<(unsigned)blocks, threads, kTable * sizeof(long long), st>>>(a, qc, n_tasks);
    else
        k_sum_terms<Four, false><<<(unsigned)n_tasks, threads, 0, st>>>(a, qc, n_tasks);
    return cudaGetLastError();
}

}  // namespace

cudaError_t sum_terms(const KsgLaunch &a, int qc, int n_groups, int n_sms, cudaStream_t st)
{
    static_assert(64 % kRowsPerWarp == 0, "tiles of up to 64 queries, a multiple of 8");
    const int64_t tasks = (int64_t)a.n_qt * n_groups;
    return a.wide ? launch_sum<uint4>(a, qc, tasks, n_sms, st) : launch_sum<uint2>(a, qc, tasks, n_sms, st);
}

}  // namespace idtx
