// screen.cu -- kernels of the learned screen (a small perceptron predicting a
// candidate's largest surrogate estimate; no counterpart in the paper).
//
// Network F -> H -> H -> 1 with ReLU; flat parameters W1[H][F], b1[H],
// W2[H][H], b2[H], w3[H], b3 (fp32 master values).  Every pass reads the
// weights rounded to bfloat16 (to nearest even) and accumulates in fp32;
// biases stay fp32.  All reductions run in a fixed order, so training is
// deterministic.
//
// A batch of 256 rows is 3.5 million FMAs, so a training step is bound by the
// latency of dependent loads and by launches.  It is two launches: the rows
// (forward, loss gradient, backward to the hidden layers: a row needs every
// weight but no other row) and the parameters (gradient sums over the rows in
// order, then Adam: a parameter needs every row but no other parameter).
// Each operand is read from global memory once per block and used from shared
// memory.  Measured on GB300, 256 rows: 8.9 us a step (rows 4.2, parameters
// 4.7) against 91 us in twelve launches of a thread per element, which read
// their operands from global memory one dependent row at a time; 32 steps and
// two shuffles of 4096 rows 4.13 -> 0.54 ms, with the same bits, and 0.39 ms
// with early launches (launch_early).  Tensor cores would not help: the sums
// are short and their order is fixed.
#include <cuda_bf16.h>
#include <cuda_pipeline.h>

#include "idtx.h"
#include "ksg_common.cuh"

namespace idtx {

namespace {

constexpr int F = IDTX_SCREEN_F;
constexpr int H = IDTX_SCREEN_H;
constexpr int P = IDTX_SCREEN_NPARAMS;
constexpr int OFF_W1 = 0, OFF_B1 = H * F, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H,
              OFF_W3 = OFF_B2 + H, OFF_B3 = OFF_W3 + H;

__device__ __forceinline__ float rounded(float v)
{
    return __bfloat162float(__float2bfloat16_rn(v));
}

// Rows of a batch: x = (feats[r] - mean) * scale with r = order[start + b] (or
// start + b), the network's output y, and with BWD the gradients of the loss at
// y (dy) and at the hidden layers' sums (d2, d1).  Squared error (quantile ==
// 0): dy = dy_scale * (y - t); pinball loss of quantile q: dy_scale * ([t < y] - q).
//
// A thread per (row, hidden unit), kRowsPerBlock rows at a time; the weights
// are rounded into shared memory by every block (20 KB from L2, less than a
// launch that would do it once).  W2 has an odd row stride, so that both its
// rows (forward) and its columns (backward) are read without bank conflicts.
constexpr int kRowsPerBlock = 4;
template <bool BWD>
__global__ void __launch_bounds__(kRowsPerBlock *H)
    k_mlp_rows(const float *params, const MlpWork w, const float *feats, const int32_t *order,
               int64_t start, int B, const float *mean, const float *scale, const float *targets,
               float dy_scale, float quantile)
{
    constexpr int kThreads = kRowsPerBlock * H;
    __shared__ float s_w1[H * (F + 1)], s_w2[H * (H + 1)], s_w3[H];
    __shared__ float s_x[kRowsPerBlock][F], s_a1[kRowsPerBlock][H], s_a2[kRowsPerBlock][H],
        s_d2[kRowsPerBlock][H], s_dy[kRowsPerBlock];
    static_assert(F % 2 == 0 && H % 2 == 0, "odd row strides");
    const int tid = threadIdx.x, r = tid / H, u = tid % H;
    auto row_of = [&](int b) -> int64_t { return order ? (int64_t)order[start + b] : start + b; };
    auto input = [&](int b) {
        return u < F && b < B ? (feats[row_of(b) * F + u] - mean[u]) * scale[u] : 0.0f;
    };
    float x = input(blockIdx.x * kRowsPerBlock + r);
    cudaGridDependencySynchronize();  // the parameters are the last step's
    cudaTriggerProgrammaticLaunchCompletion();
    const float b1 = params[OFF_B1 + u], b2 = params[OFF_B2 + u], b3 = params[OFF_B3];
#pragma unroll
    for (int i = tid; i < H * H; i += kThreads)
        s_w2[i / H * (H + 1) + i % H] = rounded(params[OFF_W2 + i]);
#pragma unroll
    for (int i = tid; i < H * F; i += kThreads)
        s_w1[i / F * (F + 1) + i % F] = rounded(params[OFF_W1 + i]);
    if (tid < H) s_w3[tid] = rounded(params[OFF_W3 + tid]);
    for (int b0 = blockIdx.x * kRowsPerBlock; b0 < B; b0 += gridDim.x * kRowsPerBlock) {
        const int b = b0 + r;
        const bool ok = b < B;
        if (u < F) {
            s_x[r][u] = x;
            if (BWD && ok) w.xn[(int64_t)b * F + u] = x;
        }
        __syncthreads();
        float z = b1;
#pragma unroll
        for (int k = 0; k < F; ++k) z = fmaf(s_w1[u * (F + 1) + k], s_x[r][k], z);
        const float a1 = fmaxf(z, 0.0f);
        s_a1[r][u] = a1;
        __syncthreads();
        z = b2;
#pragma unroll 16
        for (int k = 0; k < H; ++k) z = fmaf(s_w2[u * (H + 1) + k], s_a1[r][k], z);
        const float a2 = fmaxf(z, 0.0f);
        s_a2[r][u] = a2;
        __syncthreads();
        if (u == 0) {
            float y = b3;
#pragma unroll 16
            for (int k = 0; k < H; ++k) y = fmaf(s_w3[k], s_a2[r][k], y);
            if (ok) w.y[b] = y;
            if (BWD) {
                const float d = ok ? y - targets[row_of(b)] : 0.0f;
                const float dy = dy_scale * (quantile > 0.0f ? (d > 0.0f ? 1.0f : 0.0f) - quantile : d);
                s_dy[r] = dy;
                if (ok) w.dy[b] = dy;
            }
        }
        if (BWD) {
            __syncthreads();
            const float d2 = a2 > 0.0f ? fmaf(s_w3[u], s_dy[r], 0.0f) : 0.0f;
            s_d2[r][u] = d2;
            __syncthreads();
            float acc = 0.0f;
#pragma unroll 16
            for (int n = 0; n < H; ++n) acc = fmaf(s_w2[n * (H + 1) + u], s_d2[r][n], acc);
            if (ok) {
                const int64_t at = (int64_t)b * H + u;
                w.a1[at] = a1;
                w.a2[at] = a2;
                w.d2[at] = d2;
                w.d1[at] = a1 > 0.0f ? acc : 0.0f;
            }
        }
        x = input(b + gridDim.x * kRowsPerBlock);
        __syncthreads();  // the row's shared values are done with
    }
}

// *loss_acc += sum over the rows of (y - t)^2, or of the pinball loss (t -
// y)(q - [t < y]).  One block, fixed order.
__global__ void k_loss(const float *y, const float *targets, int64_t start, int B, float quantile,
                       double *loss_acc)
{
    __shared__ double s_part[8];
    double part = 0.0;
    for (int b = threadIdx.x; b < B; b += blockDim.x) {
        const float d = y[b] - targets[start + b];
        if (quantile > 0.0f) {
            const float below = d > 0.0f ? 1.0f : 0.0f;  // [t < y]
            part += (double)(-d) * ((double)quantile - (double)below);
        } else {
            part += (double)d * (double)d;
        }
    }
    for (int o = 16; o >= 1; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        double sum = 0.0;
        for (int t = 0; t < (int)blockDim.x / 32; ++t) sum += s_part[t];
        *loss_acc += sum;
    }
}

// Gradient of every parameter, gW[n][k] = sum over the batch's rows in order of
// dz[b][n] in[b][k] (a bias is the weight of an input of 1), then with ADAM its
// update, else the gradient written to w.grad.  A block per tile of kTileN x
// kTileK parameters of a layer, a thread per parameter; the tile's columns of
// both operands are staged kStage rows at a time.  Small tiles spread the
// staging, which is what takes the time, over more SMs.
constexpr int kTileN = 8, kTileK = 16, kStage = 256;
constexpr int kTilesK = (H + kTileK) / kTileK;          // H inputs and the bias
constexpr int kTiles2 = H / kTileN * kTilesK;           // hidden layer 2
constexpr int kTiles1 = H / kTileN;                     // hidden layer 1
constexpr int kTiles = kTiles2 + kTiles1 + kTilesK;     // and the output layer
static_assert(H % kTileN == 0 && H % kTileK == 0 && F + 1 <= kTileK, "layer tiles");

template <bool ADAM>
__global__ void __launch_bounds__(kTileN *kTileK)
    k_mlp_params(const MlpWork w, int B, float *params, float *m, float *v, float lr, float c1,
                 float c2)
{
    constexpr int kThreads = kTileN * kTileK;
    __shared__ __align__(16) float s_in[kStage * kTileK], s_dz[kStage * kTileN];
    const int tid = threadIdx.x, kk = tid % kTileK, nn = tid / kTileK;
    int t = blockIdx.x, n0, k0, K, N, off_w, off_b;
    const float *in, *dz;
    if (t < kTiles2) {
        n0 = t / kTilesK * kTileN, k0 = t % kTilesK * kTileK, K = H, N = H;
        in = w.a1, dz = w.d2, off_w = OFF_W2, off_b = OFF_B2;
    } else if (t < kTiles2 + kTiles1) {
        n0 = (t - kTiles2) * kTileN, k0 = 0, K = F, N = H;
        in = w.xn, dz = w.d1, off_w = OFF_W1, off_b = OFF_B1;
    } else {
        n0 = 0, k0 = (t - kTiles2 - kTiles1) * kTileK, K = H, N = 1;
        in = w.a2, dz = w.dy, off_w = OFF_W3, off_b = OFF_B3;
    }
    const int n = n0 + nn, k = k0 + kk;
    const bool mine = n < N && k <= K;
    const int par = k < K ? off_w + n * K + k : off_b + n;
    float p = 0.0f, mi = 0.0f, vi = 0.0f;
    if (ADAM && mine) {
        p = params[par];
        mi = m[par];
        vi = v[par];
    }
    cudaGridDependencySynchronize();  // the rows are done
    cudaTriggerProgrammaticLaunchCompletion();
    float acc = 0.0f;
    for (int b0 = 0; b0 < B; b0 += kStage) {
        const int rows = min(kStage, B - b0);
        if (K == H && k0 < H) {
            for (int i = tid; i < rows * (kTileK / 4); i += kThreads) {
                const int b = i / (kTileK / 4), c = i % (kTileK / 4) * 4;
                __pipeline_memcpy_async(s_in + b * kTileK + c, in + (int64_t)(b0 + b) * K + k0 + c, 16);
            }
        } else {
            for (int i = tid; i < rows * kTileK; i += kThreads) {
                const int b = i / kTileK, c = k0 + i % kTileK;
                if (c < K)
                    __pipeline_memcpy_async(s_in + i, in + (int64_t)(b0 + b) * K + c, 4);
                else
                    s_in[i] = c == K ? 1.0f : 0.0f;
            }
        }
        if (N == H) {
            for (int i = tid; i < rows * (kTileN / 4); i += kThreads) {
                const int b = i / (kTileN / 4), c = i % (kTileN / 4) * 4;
                __pipeline_memcpy_async(s_dz + b * kTileN + c, dz + (int64_t)(b0 + b) * H + n0 + c, 16);
            }
        } else {
            for (int b = tid; b < rows; b += kThreads)
                __pipeline_memcpy_async(s_dz + b * kTileN, dz + b0 + b, 4);
        }
        __pipeline_commit();
        __pipeline_wait_prior(0);
        __syncthreads();
        if (mine) {
#pragma unroll 16
            for (int b = 0; b < rows; ++b) acc = fmaf(s_dz[b * kTileN + nn], s_in[b * kTileK + kk], acc);
        }
        __syncthreads();
    }
    if (!mine) return;
    if (ADAM) {
        mi = 0.9f * mi + 0.1f * acc;
        vi = 0.999f * vi + 0.001f * acc * acc;
        m[par] = mi;
        v[par] = vi;
        params[par] = p - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
    } else {
        w.grad[par] = acc;
    }
}

// A launch that may start while the kernel before it in the stream still runs:
// both kernels of a training step take their operands of earlier steps, then
// wait for the other (cudaGridDependencySynchronize), and let the next one
// start only after that wait.  So what is read before a wait was complete
// when the kernel before started its own work: the rows and their order, and
// for k_mlp_params the parameters and moments of the last step.
template <typename... Args, typename... Values>
cudaError_t launch_early(void (*kernel)(Args...), int blocks, int threads, cudaStream_t st,
                         Values... values)
{
    cudaLaunchAttribute early = {};
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cfg.attrs = &early;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, Args(values)...);
}

constexpr int kMaxRowBlocks = 1024;
int row_blocks(int B)
{
    return B < kMaxRowBlocks * kRowsPerBlock ? (B + kRowsPerBlock - 1) / kRowsPerBlock
                                             : kMaxRowBlocks;
}

}  // namespace

size_t mlp_work_floats(int B) { return (size_t)B * (4 * H + F + 2) + (size_t)P; }

void mlp_work_carve(float *base, int B, MlpWork *w)
{
    float *q = base;  // the rows of H first: they are copied 16 bytes at a time
    w->a1 = q, q += (size_t)B * H;
    w->a2 = q, q += (size_t)B * H;
    w->d2 = q, q += (size_t)B * H;
    w->d1 = q, q += (size_t)B * H;
    w->xn = q, q += (size_t)B * F;
    w->y = q, q += B;
    w->dy = q, q += B;
    w->grad = q;
}

cudaError_t mlp_forward(const float *params, const MlpWork &w, const float *feats, int64_t start,
                        int B, const float *mean, const float *scale, cudaStream_t st)
{
    k_mlp_rows<false><<<row_blocks(B), kRowsPerBlock * H, 0, st>>>(
        params, w, feats, nullptr, start, B, mean, scale, nullptr, 0.0f, 0.0f);
    return cudaGetLastError();
}

cudaError_t mlp_rows(const float *params, const MlpWork &w, const float *feats,
                     const float *targets, const int32_t *order, int64_t start, int B,
                     const float *mean, const float *scale, float dy_scale, float quantile,
                     bool early, cudaStream_t st)
{
    if (early)
        return launch_early(k_mlp_rows<true>, row_blocks(B), kRowsPerBlock * H, st, params, w, feats,
                            order, start, B, mean, scale, targets, dy_scale, quantile);
    k_mlp_rows<true><<<row_blocks(B), kRowsPerBlock * H, 0, st>>>(
        params, w, feats, order, start, B, mean, scale, targets, dy_scale, quantile);
    return cudaGetLastError();
}

cudaError_t mlp_loss(const MlpWork &w, const float *targets, int64_t start, int B, float quantile,
                     double *loss_acc, cudaStream_t st)
{
    k_loss<<<1, 256, 0, st>>>(w.y, targets, start, B, quantile, loss_acc);
    return cudaGetLastError();
}

cudaError_t mlp_grad(const MlpWork &w, int B, cudaStream_t st)
{
    k_mlp_params<false><<<kTiles, kTileN * kTileK, 0, st>>>(w, B, nullptr, nullptr, nullptr, 0.0f,
                                                            1.0f, 1.0f);
    return cudaGetLastError();
}

cudaError_t mlp_adam(const MlpWork &w, int B, float *params, float *m, float *v, int step, float lr,
                     cudaStream_t st)
{
    const float c1 = 1.0f - powf(0.9f, (float)step), c2 = 1.0f - powf(0.999f, (float)step);
    return launch_early(k_mlp_params<true>, kTiles, kTileN * kTileK, st, w, B, params, m, v, lr, c1,
                        c2);
}

}  // namespace idtx
