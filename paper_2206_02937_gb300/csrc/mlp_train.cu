// mlp_train.cu -- training of the surrogate network on the GPU (arXiv
// 2206.02937, Sec. 3.2: the network is trained against the analytic
// probability with the mean absolute error loss and the Adam optimizer at
// learning rate 1e-3; Sec. 4: the implementation also allows training inside
// the simulation).
//
// One training step over a minibatch of n samples (inputs u, k; targets y;
// per-sample weights w from the data balancing) is two launches:
//   k_train_f32 or (tensor-core precision) k_train_tc of mlp_train_tc.cu
//                    forward and backward over tiles of samples; the gradient
//                    sums, the loss numerator and the weight sum are added to
//                    MlpDev::acc;
//   k_mlp_finish     (mlp.cu) Adam (Kingma and Ba 2014, Algorithm 1) on the
//                    FP32 master parameters with the gradient divided by sum
//                    w, the inference images rebuilt, acc cleared for the
//                    next step.
#include "ctx.hpp"
#include "device_math.cuh"
#include "features.cuh"

namespace compton {
namespace {

__device__ __forceinline__ float sigm(float z) { return 1.0f / (1.0f + expf(-z)); }

struct TrainArgs {
    MlpDev m;
    const float* u[3];
    const float* k[3];
    const float* y;
    const float* w;  // nullable: all ones
    int64_t n;
};

// ---------------------------------------------------------------------------
// FP32 gradient on the CUDA cores.  One CTA per SM takes tiles of 64 samples;
// every contraction of the tile (z = a W^T, dX = delta W, dW = delta^T a, each
// 64 x 64 x 64) is a register tile of 4 x 4 outputs per thread over operands in
// shared memory: two 16-byte shared loads per 16 multiply-adds, where one
// sample per thread took 16 such loads for 64 and left an SM eight warps.
// Activations and deltas lie as [unit][sample] rows 68 words apart, so that the
// 16-byte loads along the samples of neighbouring rows (dW) fall into different
// banks; the weights lie in both orders.  Pre-activations never leave the
// thread: the backward pass uses the same thread-to-output map as the forward
// pass, so the derivative of SiLU stays in 16 registers per layer, and dW is
// accumulated over the CTA's tiles in registers (a tile's sums first, then
// added, so that no FP32 sum is longer than a tile plus the tiles).
//
// What bounds it: the FP32 pipe (9.2 contractions of 1.1 us each per tile) and
// the SiLU's exact exponentials and divisions.
// ---------------------------------------------------------------------------
constexpr int kTrThreads = 256;
constexpr int kTrTile = 64;              // samples per tile
constexpr int kTrStride = kTrTile + 4;   // words between rows of activations and deltas
constexpr int kTrMat = 64 * kTrStride;   // one 64-row block of activations
struct TrainSmem {
    static constexpr int wt = 0;                       // W_1..W_3 as [in][out]
    static constexpr int wj = wt + 3 * 4096;           // W_1..W_3 as [out][in]
    static constexpr int wt0 = wj + 3 * 4096;          // W_0 as [in][out], 6 rows
    static constexpr int bias = wt0 + 6 * 64;          // 4 x 64
    static constexpr int w4 = bias + 256;              // 64
    static constexpr int feat = w4 + 64;               // 6 rows
    static constexpr int act = feat + 6 * kTrStride;   // a_0..a_3
    static constexpr int delta = act + 4 * kTrMat;     // two blocks of deltas
    static constexpr int dout = delta + 2 * kTrMat;    // delta of the output unit per sample
    static constexpr int words = dout + kTrTile;
};

__device__ __forceinline__ void cp_async16(float* smem_dst, const float* gmem_src)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(gmem_src) : "memory");
}

// acc[p][q] += x[p] y[q]
__device__ __forceinline__ void outer4(float (&acc)[4][4], float4 x, float4 y)
{
    const float xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(xv[p], yv[q], acc[p][q]);
}

__device__ __forceinline__ float dot4(float4 x, float4 y, float t)
{
    return fmaf(x.w, y.w, fmaf(x.z, y.z, fmaf(x.y, y.y, fmaf(x.x, y.x, t))));
}

__global__ void __launch_bounds__(kTrThreads, 1) k_train_f32(TrainArgs a)
{
    chain_start();
    extern __shared__ __align__(16) float sm[];
    using S = TrainSmem;
    const int tid = threadIdx.x;
    const MlpDev& m = a.m;
    // forward operands first, the backward pass's weight order behind them
    for (int i = tid; i < 3 * 1024; i += kTrThreads) cp_async16(sm + S::wt + 4 * i, m.wt32 + 4096 + 4 * i);
    if (tid < 6 * 16) cp_async16(sm + S::wt0 + 4 * tid, m.wt32 + 4 * tid);
    if (tid < 64) cp_async16(sm + S::bias + 4 * tid, m.bias + 4 * tid);
    if (tid < 16) cp_async16(sm + S::w4 + 4 * tid, m.w4 + 4 * tid);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    for (int l = 1; l < 4; ++l)
        for (int i = tid; i < 1024; i += kTrThreads)
            cp_async16(sm + S::wj + (l - 1) * 4096 + 4 * i, m.theta + mlp_off_w(l) + 4 * i);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    const float b4 = m.b4[0];

    const int s0 = 4 * (tid & 15), j0 = 4 * (tid >> 4);  // forward and dX: samples s0.., units j0..
    const int di = tid & 15, dj = tid >> 4;              // dW: inputs di + 16 q, outputs dj + 16 p
    const int bj = tid >> 2, bp = tid & 3;               // bias sums: unit bj, a quarter of the samples
    float dw[3][4][4], db[4] = {0, 0, 0, 0}, dw0[3] = {0, 0, 0}, dw4 = 0.0f, db4 = 0.0f;
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) dw[l][p][q] = 0.0f;
    float loss_num = 0.0f, wsum = 0.0f;

    for (int64_t base = (int64_t)blockIdx.x * kTrTile; base < a.n; base += (int64_t)gridDim.x * kTrTile) {
        const int ns = a.n - base < kTrTile ? (int)(a.n - base) : kTrTile;
        // ---- features ----
        if (tid < kTrTile) {
            float f[6] = {0, 0, 0, 0, 0, 0};
            if (tid < ns) {
                const int64_t s = base + tid;
                features(m, a.u[0][s], a.u[1][s], a.u[2][s], a.k[0][s], a.k[1][s], a.k[2][s], f);
            }
#pragma unroll
            for (int i = 0; i < 6; ++i) sm[S::feat + i * kTrStride + tid] = f[i];
        }
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        __syncthreads();
        // ---- forward ----
        float ds[4][4][4];  // SiLU'(z_l) of units j0.., samples s0..
#pragma unroll
        for (int l = 0; l < 4; ++l) {
            float z[4][4];
#pragma unroll
            for (int p = 0; p < 4; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q) z[p][q] = sm[S::bias + 64 * l + j0 + p];
            const float* in = l == 0 ? sm + S::feat : sm + S::act + (l - 1) * kTrMat;
            const float* w = l == 0 ? sm + S::wt0 : sm + S::wt + (l - 1) * 4096;
#pragma unroll 8
            for (int i = 0; i < (l == 0 ? 6 : 64); ++i)
                outer4(z, *reinterpret_cast<const float4*>(w + 64 * i + j0),
                       *reinterpret_cast<const float4*>(in + kTrStride * i + s0));
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                float h[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float zz = z[p][q], sg = sigm(zz);
                    ds[l][p][q] = sg * (1.0f + zz * (1.0f - sg));
                    h[q] = zz * sg;
                    if (s0 + q >= ns) h[q] = ds[l][p][q] = 0.0f;
                }
                *reinterpret_cast<float4*>(sm + S::act + l * kTrMat + (j0 + p) * kTrStride + s0) =
                    make_float4(h[0], h[1], h[2], h[3]);
            }
            __syncthreads();
        }
        // ---- output, loss and the output unit's delta: one thread per sample ----
        if (tid < kTrTile) {
            float d_out = 0.0f;
            if (tid < ns) {
                float zo = b4;
#pragma unroll 16
                for (int j = 0; j < 64; ++j) zo = fmaf(sm[S::act + 3 * kTrMat + j * kTrStride + tid], sm[S::w4 + j], zo);
                const float yp = sigm(zo);
                const float wi = a.w ? a.w[base + tid] : 1.0f;
                const float diff = yp - a.y[base + tid];
                loss_num += wi * fabsf(diff);
                wsum += wi;
                // unnormalised: the 1 / sum w factor is applied in Adam
                const float g = diff > 0.0f ? wi : (diff < 0.0f ? -wi : 0.0f);
                d_out = g * yp * (1.0f - yp);
            }
            sm[S::dout + tid] = d_out;
            db4 += d_out;
        }
        asm volatile("cp.async.wait_group 0;\n" ::: "memory");
        __syncthreads();
        // ---- backward ----
        {
            const float4 d4 = *reinterpret_cast<const float4*>(sm + S::dout + s0);
            const float d[4] = {d4.x, d4.y, d4.z, d4.w};
#pragma unroll
            for (int p = 0; p < 4; ++p) {
                const float w = sm[S::w4 + j0 + p];
                *reinterpret_cast<float4*>(sm + S::delta + (j0 + p) * kTrStride + s0) =
                    make_float4(w * d[0] * ds[3][p][0], w * d[1] * ds[3][p][1], w * d[2] * ds[3][p][2],
                                w * d[3] * ds[3][p][3]);
            }
            // dw_4
            const float4* av = reinterpret_cast<const float4*>(sm + S::act + 3 * kTrMat + bj * kTrStride + 16 * bp);
            const float4* dv = reinterpret_cast<const float4*>(sm + S::dout + 16 * bp);
            float t = 0.0f;
#pragma unroll
            for (int i = 0; i < 4; ++i) t = dot4(av[i], dv[i], t);
            dw4 += t;
        }
        __syncthreads();
#pragma unroll
        for (int l = 3; l >= 0; --l) {
            const float* dl = sm + S::delta + ((3 - l) & 1) * kTrMat;
            if (l > 0) {
                // delta_{l-1} = (delta_l W_l) SiLU'(z_{l-1}), units j0.. of layer l - 1
                float t[4][4] = {};
#pragma unroll 8
                for (int j = 0; j < 64; ++j)
                    outer4(t, *reinterpret_cast<const float4*>(sm + S::wj + (l - 1) * 4096 + 64 * j + j0),
                           *reinterpret_cast<const float4*>(dl + kTrStride * j + s0));
                float* dn = sm + S::delta + ((4 - l) & 1) * kTrMat;
#pragma unroll
                for (int p = 0; p < 4; ++p)
                    *reinterpret_cast<float4*>(dn + (j0 + p) * kTrStride + s0) =
                        make_float4(t[p][0] * ds[l - 1][p][0], t[p][1] * ds[l - 1][p][1], t[p][2] * ds[l - 1][p][2],
                                    t[p][3] * ds[l - 1][p][3]);
                // dW_l
                const float* in = sm + S::act + (l - 1) * kTrMat;
                float g[4][4] = {};
#pragma unroll 2
                for (int s = 0; s < kTrTile; s += 4) {
                    float4 dv[4], av[4];
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        dv[p] = *reinterpret_cast<const float4*>(dl + (dj + 16 * p) * kTrStride + s);
                        av[p] = *reinterpret_cast<const float4*>(in + (di + 16 * p) * kTrStride + s);
                    }
#pragma unroll
                    for (int p = 0; p < 4; ++p)
#pragma unroll
                        for (int q = 0; q < 4; ++q) g[p][q] = dot4(dv[p], av[q], g[p][q]);
                }
#pragma unroll
                for (int p = 0; p < 4; ++p)
#pragma unroll
                    for (int q = 0; q < 4; ++q) dw[l - 1][p][q] += g[p][q];
            } else if (tid < 128) {
                // dW_0: output tid / 2, three of the six inputs
                float g[3] = {0, 0, 0};
                for (int s = 0; s < kTrTile; s += 4) {
                    const float4 dv = *reinterpret_cast<const float4*>(dl + (tid >> 1) * kTrStride + s);
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        g[q] = dot4(dv, *reinterpret_cast<const float4*>(sm + S::feat + (3 * (tid & 1) + q) * kTrStride + s),
                                    g[q]);
                }
#pragma unroll
                for (int q = 0; q < 3; ++q) dw0[q] += g[q];
            }
            {
                const float4* dv = reinterpret_cast<const float4*>(dl + bj * kTrStride + 16 * bp);
                float t = 0.0f;
#pragma unroll
                for (int i = 0; i < 4; ++i) t += (dv[i].x + dv[i].y) + (dv[i].z + dv[i].w);
                db[l] += t;
            }
            __syncthreads();
        }
    }

    // ---- the CTA's sums into the step's accumulators ----
    float* acc = m.acc;
#pragma unroll
    for (int l = 1; l < 4; ++l)
#pragma unroll
        for (int p = 0; p < 4; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                atomicAdd(&acc[mlp_off_w(l) + (dj + 16 * p) * 64 + di + 16 * q], dw[l - 1][p][q]);
    if (tid < 128)
#pragma unroll
        for (int q = 0; q < 3; ++q) atomicAdd(&acc[(tid >> 1) * 6 + 3 * (tid & 1) + q], dw0[q]);
#pragma unroll
    for (int l = 0; l < 5; ++l) {
        float t = l < 4 ? db[l] : dw4;
        t += __shfl_xor_sync(0xffffffffu, t, 1);
        t += __shfl_xor_sync(0xffffffffu, t, 2);
        if (bp == 0) atomicAdd(&acc[(l < 4 ? mlp_off_b(l) : mlp_off_w(4)) + bj], t);
    }
    if (tid < kTrTile) {
        for (int d = 16; d > 0; d >>= 1) {
            loss_num += __shfl_xor_sync(0xffffffffu, loss_num, d);
            wsum += __shfl_xor_sync(0xffffffffu, wsum, d);
            db4 += __shfl_xor_sync(0xffffffffu, db4, d);
        }
        if ((tid & 31) == 0) {
            atomicAdd(&acc[mlp_off_b(4)], db4);
            atomicAdd(&m.acc_loss[0], (double)loss_num);
            atomicAdd(&m.acc_loss[1], (double)wsum);
        }
    }
}

// Data balancing (Sec. 3.2: events of every probability range should appear
// about equally often).  Sample i belongs to bin b = number of inner edges
// <= r_i; its weight is n / (count_b * number of non-empty bins).
constexpr int kMaxBalanceBins = 256;

__device__ __forceinline__ int balance_bin(const float* inner, int n_inner, float r)
{
    int lo = 0, hi = n_inner;  // first inner edge > r
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (inner[mid] <= r) lo = mid + 1; else hi = mid;
    }
    return lo;
}

__global__ void k_balance_hist(const float* __restrict__ r, int64_t n, const float* __restrict__ edges, int n_bins,
                               int* __restrict__ count)
{
    __shared__ float inner[kMaxBalanceBins];
    __shared__ int h[kMaxBalanceBins];
    for (int i = threadIdx.x; i < n_bins; i += blockDim.x) {
        h[i] = 0;
        if (i < n_bins - 1) inner[i] = edges[i + 1];
    }
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        atomicAdd(&h[balance_bin(inner, n_bins - 1, r[i])], 1);
    __syncthreads();
    for (int i = threadIdx.x; i < n_bins; i += blockDim.x)
        if (h[i]) atomicAdd(&count[i], h[i]);
}

__global__ void k_balance_weights(const float* __restrict__ r, int64_t n, const float* __restrict__ edges,
                                  int n_bins, const int* __restrict__ count, float* __restrict__ w)
{
    __shared__ float inner[kMaxBalanceBins];
    __shared__ float inv[kMaxBalanceBins];
    __shared__ int nonempty;
    if (threadIdx.x == 0) {
        int ne = 0;
        for (int i = 0; i < n_bins; ++i) ne += count[i] > 0;
        nonempty = ne;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n_bins; i += blockDim.x) {
        if (i < n_bins - 1) inner[i] = edges[i + 1];
        inv[i] = count[i] > 0 ? (float)((double)n / ((double)count[i] * (double)nonempty)) : 0.0f;
    }
    __syncthreads();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        w[i] = inv[balance_bin(inner, n_bins - 1, r[i])];
}

}  // namespace

compton_status launch_balance_weights(compton_ctx* ctx, const float* r, int64_t n, const float* edges_host,
                                      int n_bins, float* w_out, cudaStream_t stream)
{
    if (n_bins < 1 || n_bins > kMaxBalanceBins) return COMPTON_EINVAL;
    COMPTON_CUDA_TRY(ctx, cudaMemcpyAsync(ctx->mlp.edges, edges_host, sizeof(float) * (n_bins + 1),
                                          cudaMemcpyHostToDevice, stream));
    COMPTON_CUDA_TRY(ctx, cudaMemsetAsync(ctx->mlp.hist, 0, sizeof(int) * n_bins, stream));
    int64_t blocks = (n + 255) / 256;
    if (blocks > (int64_t)ctx->n_sm * 8) blocks = (int64_t)ctx->n_sm * 8;
    k_balance_hist<<<(unsigned)blocks, 256, 0, stream>>>(r, n, ctx->mlp.edges, n_bins, ctx->mlp.hist);
    COMPTON_LAUNCH_CHECK(ctx, "k_balance_hist");
    k_balance_weights<<<(unsigned)blocks, 256, 0, stream>>>(r, n, ctx->mlp.edges, n_bins, ctx->mlp.hist, w_out);
    COMPTON_LAUNCH_CHECK(ctx, "k_balance_weights");
    return COMPTON_OK;
}

compton_status launch_mlp_train_step(compton_ctx* ctx, const float* ux, const float* uy, const float* uz,
                                     const float* kx, const float* ky, const float* kz, const float* y,
                                     const float* w, int64_t n, float lr, cudaStream_t stream)
{
    // the accumulators are zero between steps (k_mlp_finish clears them); after
    // a step that failed between its two launches they are cleared here
    if (ctx->train_dirty)
        COMPTON_CUDA_TRY(ctx, cudaMemsetAsync(ctx->mlp.acc, 0, kMlpAccBytes, stream));
    ctx->train_dirty = true;
    compton_status st;
    if (ctx->train_tc) {
        st = launch_mlp_grad_tc(ctx, ux, uy, uz, kx, ky, kz, y, w, n, stream);
        if (st != COMPTON_OK) return st;
    } else {
        TrainArgs a;
        a.m = ctx->mlp;
        a.u[0] = ux;
        a.u[1] = uy;
        a.u[2] = uz;
        a.k[0] = kx;
        a.k[1] = ky;
        a.k[2] = kz;
        a.y = y;
        a.w = w;
        a.n = n;
        const int smem = TrainSmem::words * (int)sizeof(float);
        COMPTON_CUDA_TRY(ctx, cudaFuncSetAttribute(k_train_f32, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
        const int64_t tiles = (n + kTrTile - 1) / kTrTile;
        const unsigned grid = (unsigned)(tiles < ctx->n_sm ? tiles : ctx->n_sm);
        launch_chained(k_train_f32, grid, kTrThreads, smem, stream, a);
        COMPTON_LAUNCH_CHECK(ctx, "k_train_f32");
    }
    st = mlp_adam(ctx, lr, stream);
    if (st == COMPTON_OK) ctx->train_dirty = false;
    return st;
}

}  // namespace compton
