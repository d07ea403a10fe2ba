// sums.cu -- the digamma terms of the list kernel's counts and their sums.
#include <cuda_runtime.h>

#include "ksg_common.cuh"

namespace idtx {

namespace {

// The digamma terms of a query tile of one group, a lane per job, summed in
// the tile kernel's order: warp w of the block's nws sums over the queries m =
// w, w + nws, ..., and the first adds those sums in order of w.  (One warp for
// the whole tile took 18 us at N = 1000, where few tiles meet many SMs.)
__global__ void k_sum_terms(const KsgLaunch a, int qc)
{
    __shared__ double s_sum[32][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nws = blockDim.x >> 5;
    const int qt = blockIdx.x, grp = blockIdx.y;
    const int job = grp * 32 + lane;
    const bool job_ok = job < a.n_jobs;
    const int64_t q0 = (int64_t)qt * qc;
    unsigned sz = 0, syz = 0;  // for the work counters
    constexpr int kRows = 8;   // rows in flight
    double tsum = 0.0;
    for (int m0 = w; m0 < qc; m0 += nws * kRows) {
        int z[kRows], xz[kRows], yz[kRows];
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            const int m = m0 + u * nws;
            const bool in = m < qc && q0 + m < a.n;
            const int64_t at = ((int64_t)grp * a.n_pad + (in ? q0 + m : q0)) * 32 + lane;
            z[u] = in ? (int)__ldcs(a.cz + at) : -1;
            xz[u] = __ldcs(a.cxz + at);
            yz[u] = __ldcs(a.cyz + at);
        }
#pragma unroll
        for (int u = 0; u < kRows; ++u) {
            if (z[u] < 0 || !job_ok) continue;
            sz += z[u];
            syz += yz[u];
            tsum += __ldg(a.psi + z[u] + 1) - __ldg(a.psi + xz[u] + 1) - __ldg(a.psi + yz[u] + 1);
            if (a.cnt_out) {
                const int64_t qi = q0 + m0 + u * nws;
                const int64_t orig = a.order ? (int64_t)a.order[qi] : qi;
                int32_t *co = a.cnt_out + (int64_t)job * 3 * a.n;
                co[orig] = xz[u];
                co[a.n + orig] = yz[u];
                co[2 * a.n + orig] = z[u];
            }
        }
    }
    s_sum[w][lane] = tsum;
    if (a.work) {
        sz = __reduce_add_sync(0xffffffffu, sz);
        syz = __reduce_add_sync(0xffffffffu, syz);
        if (lane < 2) atomicAdd(&a.work[8 + lane], (unsigned long long)(lane ? syz : sz));
    }
    __syncthreads();
    if (w == 0 && job_ok) {
        double s = 0.0;
        for (int v = 0; v < nws; ++v) s += s_sum[v][lane];
        a.partial[(int64_t)job * a.n_qt + qt] = s;
    }
}

}  // namespace

cudaError_t sum_terms(const KsgLaunch &a, int qc, int nws, int n_groups, cudaStream_t st)
{
    k_sum_terms<<<dim3((unsigned)a.n_qt, (unsigned)n_groups), nws * 32, 0, st>>>(a, qc);
    return cudaGetLastError();
}

}  // namespace idtx
