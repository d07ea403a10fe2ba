// sums.cu -- the digamma terms of the list kernel's counts and their sums.
#include <cuda_runtime.h>

#include "ksg_common.cuh"

namespace idtx {

namespace {

// A tile of qc queries of one group.  A lane takes four jobs of a query (8
// lanes a query, four queries a warp), so its counts come in 8-byte loads, two
// queries' in flight; the lanes' and warps' sums are added at the end.
// Bound by the table lookups (the counts are 6 bytes a query and job).  N = 9995, 9447
// estimates: 0.58 -> 0.30 ms against terms and sums in fp64, of which an SM
// does two operations a clock (see digamma_sum).
constexpr int kRowsPerWarp = 8;
template <typename Four>  // four counts: uint2 of 16 bits each, uint4 of 32
__global__ void k_sum_terms(const KsgLaunch a, int qc)
{
    __shared__ long long s_sum[32][32];  // [warp][job]
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const int qt = blockIdx.x, grp = blockIdx.y;
    const int j0 = (lane & 7) * 4, n_job = min(4, a.n_jobs - (grp * 32 + j0));
    const int64_t q0 = (int64_t)qt * qc;
    unsigned sz = 0, syz = 0;  // for the work counters
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
            sum[t] += __ldg(a.psi + nz + 1) - __ldg(a.psi + nxz + 1) - __ldg(a.psi + nyz + 1);
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
    if (a.work) {
        sz = __reduce_add_sync(0xffffffffu, sz);
        syz = __reduce_add_sync(0xffffffffu, syz);
        if (lane < 2) atomicAdd(&a.work[8 + lane], (unsigned long long)(lane ? syz : sz));
    }
    __syncthreads();
    const int job = grp * 32 + lane;
    if (w == 0 && job < a.n_jobs) {
        long long s = 0;
        for (int v = 0; v < nw; ++v) s += s_sum[v][lane];
        a.partial[(int64_t)job * a.n_qt + qt] = digamma_sum(s);
    }
}

}  // namespace

cudaError_t sum_terms(const KsgLaunch &a, int qc, int n_groups, cudaStream_t st)
{
    static_assert(64 % kRowsPerWarp == 0, "tiles of up to 64 queries, a multiple of 8");
    const dim3 grid((unsigned)a.n_qt, (unsigned)n_groups);
    const unsigned threads = (unsigned)(qc / kRowsPerWarp * 32);
    if (a.wide)
        k_sum_terms<uint4><<<grid, threads, 0, st>>>(a, qc);
    else
        k_sum_terms<uint2><<<grid, threads, 0, st>>>(a, qc);
    return cudaGetLastError();
}

}  // namespace idtx
