// pnet.cu -- the paper's own surrogate network (arXiv 2206.02937, Sec. 3.2:
// three hidden layers of 9, 12 and 9 ReLU units, one sigmoid output, trained
// with the mean absolute error and Adam).
//
// Inputs (Fig. 2a: both momenta, both macro-particle weights and the cell's
// maximum probability): f = [sgnlog(u/s_u)/n_u (3), sgnlog(k/s_k)/n_k (3),
// ln(w_e)/8, ln(w_g)/8, ln(P_max)/8] with P_max = 2 n dt; output
// r = sigma_KN v / (2 sigma_T) (the probability over P_max).  337
// parameters, W0 (9x9) b0 W1 (12x9) b1 W2 (9x12) b2 W3 (1x9) b3, each W
// (out, in) row-major.
//
// The network is tiny (306 multiply-adds per sample), so everything runs on
// the CUDA cores in FP32, one sample per thread, with the parameters staged
// in shared memory:
//   k_pnet_infer   r per explicit pair, or -- in the surrogate step -- per
//                  candidate of the candidate list (weights w/V of the pair's
//                  particles, P_max = 2 n_p dt of the pair) with the decision
//                  made in the same thread (analytic probability outside the
//                  training range) and accepted pairs appended to the list;
//   k_pnet_train   one training step: forward and backward per sample, the
//                  parameters' gradients as products of rows staged in shared
//                  memory, and Adam by the block that finishes last.
#include "ctx.hpp"
#include "device_math.cuh"
#include "features.cuh"

namespace compton {
namespace {

constexpr int kPnetThreads = 256;
constexpr int kP_W0 = 0, kP_B0 = 81, kP_W1 = 90, kP_B1 = 198, kP_W2 = 210, kP_B2 = 318, kP_W3 = 327, kP_B3 = 336;
static_assert(kP_B3 + 1 == kPnetParams, "layout");

struct PnetArgs {
    PnetDev p;
    const float* u[3];
    const float* k[3];
    int64_t n;
    float ln_we, ln_wg, ln_pmax;  // scalar inputs of explicit rows (ln of w_e, w_g, P_max)
    float* r_out;
    // candidate rows (surrogate step): the candidate list and its decision
    const CandPair* cand;
    const uint32_t* n_cand;
    float dt, gamma64, ln_w;
    const float* w_e;  // per-particle weights of the sorted species (nullptr: ln_w)
    const float* w_g;
    float* prob_out;
    uint8_t* flag_out;
    AcceptedPair* accepted;
    uint32_t* n_accepted;
    DeviceStats* stats;
    MlpDev range;  // training range (range_* fields)
    // training
    const float* y;
    const float* wts;
};

__device__ __forceinline__ void pnet_features(const PnetDev& p, const float* q, float lwe, float lwg, float lpm,
                                              float* f)
{
    const float iu = __fdividef(1.0f, p.fs[0]), nu = __fdividef(1.0f, p.fs[1]);
    const float ik = __fdividef(1.0f, p.fs[2]), nk = __fdividef(1.0f, p.fs[3]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        f[i] = sgnlog(q[i] * iu) * nu;
        f[3 + i] = sgnlog(q[3 + i] * ik) * nk;
    }
    f[6] = lwe * 0.125f;
    f[7] = lwg * 0.125f;
    f[8] = lpm * 0.125f;
}

// Forward pass; keeps the hidden activations for the backward pass.
__device__ __forceinline__ float pnet_forward(const float* th, const float* f, float* h1, float* h2, float* h3)
{
#pragma unroll
    for (int o = 0; o < 9; ++o) {
        float z = th[kP_B0 + o];
#pragma unroll
        for (int i = 0; i < 9; ++i) z = fmaf(th[kP_W0 + 9 * o + i], f[i], z);
        h1[o] = fmaxf(z, 0.0f);
    }
#pragma unroll
    for (int o = 0; o < 12; ++o) {
        float z = th[kP_B1 + o];
#pragma unroll
        for (int i = 0; i < 9; ++i) z = fmaf(th[kP_W1 + 9 * o + i], h1[i], z);
        h2[o] = fmaxf(z, 0.0f);
    }
#pragma unroll
    for (int o = 0; o < 9; ++o) {
        float z = th[kP_B2 + o];
#pragma unroll
        for (int i = 0; i < 12; ++i) z = fmaf(th[kP_W2 + 12 * o + i], h2[i], z);
        h3[o] = fmaxf(z, 0.0f);
    }
    float z = th[kP_B3];
#pragma unroll
    for (int i = 0; i < 9; ++i) z = fmaf(th[kP_W3 + i], h3[i], z);
    return __fdividef(1.0f, 1.0f + __expf(-z));
}

__device__ __forceinline__ void stage_params(const PnetDev& p, float* th)
{
    for (int i = threadIdx.x; i < kPnetParams; i += blockDim.x) th[i] = p.theta[i];
    __syncthreads();
}

// kCand: rows are candidates, decided here; else explicit rows, r written.
template <bool kCand>
__global__ void __launch_bounds__(kPnetThreads, 3) k_pnet_infer(PnetArgs a)
{
    chain_start();
    __shared__ float th[kPnetParams];
    stage_params(a.p, th);
    const unsigned lane = threadIdx.x & 31u;
    const int64_t n = kCand ? (int64_t)*a.n_cand : a.n;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // warp-uniform trip count, so the ballots see whole warps
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
    unsigned n_hit = 0, n_fb = 0;
    for (int64_t base = first; base < n; base += stride) {
        const int64_t row = base + lane;
        const bool live = row < n;
        float q[6] = {0, 0, 0, 0, 0, 0};
        CandPair c{};
        if (live) {
            if (kCand) {
                c = a.cand[row];
                q[0] = c.u[0];
                q[1] = c.u[1];
                q[2] = c.u[2];
                q[3] = c.k[0];
                q[4] = c.k[1];
                q[5] = c.k[2];
            } else {
                q[0] = a.u[0][row];
                q[1] = a.u[1][row];
                q[2] = a.u[2][row];
                q[3] = a.k[0][row];
                q[4] = a.k[1][row];
                q[5] = a.k[2][row];
            }
        }
        float f[9], h1[9], h2[12], h3[9];
        const float lpm = kCand ? logf(fmaxf(2.0f * c.dens * a.dt, 1e-30f)) : a.ln_pmax;
        float lwe = kCand ? a.ln_w : a.ln_we, lwg = kCand ? a.ln_w : a.ln_wg;
        if (kCand && live) {
            if (a.w_e) lwe = logf(a.w_e[c.ie]);
            if (a.w_g) lwg = logf(a.w_g[c.ig]);
        }
        pnet_features(a.p, q, lwe, lwg, lpm, f);
        const float r = pnet_forward(th, f, h1, h2, h3);
        if (!kCand) {
            if (live) a.r_out[row] = r;
            continue;
        }
        bool hit = false, fb = false;
        float x = -1.0f;
        if (live) {
            const float g2 = fmaf(q[0], q[0], fmaf(q[1], q[1], fmaf(q[2], q[2], 1.0f)));
            const float e2 = fmaf(q[3], q[3], fmaf(q[4], q[4], q[5] * q[5]));
            float P;
            if (mlp_in_range(a.range, g2, e2)) {
                P = one_minus_exp_neg(2.0f * c.dens * a.dt * r);
            } else {
                fb = true;
                P = analytic_prob(q[0], q[1], q[2], q[3], q[4], q[5], c.dens, a.dt, a.gamma64, &x);
            }
            hit = c.u0 < P;
            if (a.prob_out) a.prob_out[c.p] = P;
            if (a.flag_out) a.flag_out[c.p] = hit ? 1 : 0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (fb) ++n_fb;
        if (m) {
            uint32_t at = 0;
            if (lane == 0) at = atomicAdd(a.n_accepted, (uint32_t)__popc(m));
            at = __shfl_sync(0xffffffffu, at, 0);
            if (hit) {
                a.accepted[at + __popc(m & ((1u << lane) - 1u))] =
                    AcceptedPair{c.ie, c.ig, x, c.p, {q[0], q[1], q[2]}, {q[3], q[4], q[5]}, {0u, 0u}};
                ++n_hit;
            }
        }
    }
    if (kCand) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            n_hit += __shfl_xor_sync(0xffffffffu, n_hit, d);
            n_fb += __shfl_xor_sync(0xffffffffu, n_fb, d);
        }
        if (lane == 0) {
            if (n_hit) atomicAdd(&a.stats->scatters, (unsigned long long)n_hit);
            if (n_fb) atomicAdd(&a.stats->mlp_fallbacks, (unsigned long long)n_fb);
        }
    }
}

// Training step: gradient, loss and Adam in one launch.
//
// A tile of kS samples per pass: one thread per sample runs the forward and
// backward passes and leaves the sample's 70 vector components (inputs, hidden
// activations, deltas) as rows of shared memory; then every parameter's
// gradient is a dot product of two of those rows over the tile, one thread per
// parameter (the loss and the weight sum are two more such sums), so nothing
// is reduced by shuffles and no two threads add to the same word.  The rows
// are kS + 4 words apart: the eight lanes of a 16-byte shared load read
// neighbouring rows, which then lie in different banks.  A tile's sums are
// added to the thread's running sums once (two levels, as short as the tile).
// Each block adds its sums to acc; the block that finishes last (a ticket)
// takes them as the step's gradient, runs Adam and clears acc and the ticket
// for the next step, so a step needs no memset and no second launch.
//
// What bounds it: at a minibatch of 8192 the latency of one tile's chain (about
// 600 dependent multiply-adds, then 16 steps of the row products).
constexpr int kTrainSums = kPnetParams + 2;  // gradients, weighted |error| sum, weight sum
constexpr int kTrainThreads = 352;           // a thread per sum, whole warps
constexpr int kRowF = 0, kRowH1 = 9, kRowH2 = 18, kRowH3 = 30, kRowD0 = 39, kRowD1 = 48, kRowD2 = 60, kRowD3 = 69,
              kRowLoss = 70, kRowW = 71, kRowOne = 72, kTrainRows = 73;
static_assert(kTrainSums <= kTrainThreads, "a thread per sum");

// The two rows whose product sums to entry p of acc.
__device__ __forceinline__ void train_rows(int p, int& ra, int& rb)
{
    rb = kRowOne;
    if (p < kP_B0) { ra = kRowD0 + p / 9; rb = kRowF + p % 9; }
    else if (p < kP_W1) ra = kRowD0 + (p - kP_B0);
    else if (p < kP_B1) { ra = kRowD1 + (p - kP_W1) / 9; rb = kRowH1 + (p - kP_W1) % 9; }
    else if (p < kP_W2) ra = kRowD1 + (p - kP_B1);
    else if (p < kP_B2) { ra = kRowD2 + (p - kP_W2) / 12; rb = kRowH2 + (p - kP_W2) % 12; }
    else if (p < kP_W3) ra = kRowD2 + (p - kP_B2);
    else if (p < kP_B3) { ra = kRowD3; rb = kRowH3 + (p - kP_W3); }
    else if (p == kP_B3) ra = kRowD3;
    else ra = p == kPnetParams ? kRowLoss : kRowW;
}

template <int kS>
__global__ void __launch_bounds__(kTrainThreads, 1) k_pnet_train(PnetArgs a, float lr, float b1t, float b2t)
{
    chain_start();
    constexpr int kStride = kS + 4;
    extern __shared__ __align__(16) float rows[];  // [kTrainRows][kStride]
    __shared__ float th[kPnetParams];
    __shared__ bool last;
    const int tid = threadIdx.x;
    for (int i = tid; i < kS; i += kTrainThreads) rows[kRowOne * kStride + i] = 1.0f;
    stage_params(a.p, th);
    int ra = 0, rb = 0;
    if (tid < kTrainSums) train_rows(tid, ra, rb);
    const float4* va = reinterpret_cast<const float4*>(rows + ra * kStride);
    const float4* vb = reinterpret_cast<const float4*>(rows + rb * kStride);
    float sum = 0.0f;
    for (int64_t base = (int64_t)blockIdx.x * kS; base < a.n; base += (int64_t)gridDim.x * kS) {
        if (tid < kS) {
            const int64_t s = base + tid;
            float q[6] = {0, 0, 0, 0, 0, 0};
            float y = 0.0f, wt = 0.0f;
            if (s < a.n) {
                q[0] = a.u[0][s];
                q[1] = a.u[1][s];
                q[2] = a.u[2][s];
                q[3] = a.k[0][s];
                q[4] = a.k[1][s];
                q[5] = a.k[2][s];
                y = a.y[s];
                wt = a.wts ? a.wts[s] : 1.0f;
            }
            float* col = rows + tid;
            auto put = [&](int r, float v) { col[r * kStride] = v; };
            float f[9], h1[9], h2[12], h3[9];
            pnet_features(a.p, q, a.ln_we, a.ln_wg, a.ln_pmax, f);
            const float yp = pnet_forward(th, f, h1, h2, h3);
            // the weights are read from shared memory again in the backward
            // pass (kept in registers they spill)
            asm volatile("" ::: "memory");
            const float err = yp - y;
            put(kRowLoss, wt * fabsf(err));
            put(kRowW, wt);
            // d loss / d z of the output times sum w: w sign(err) sigma'(z)
            // (Adam divides by the weight sum)
            const float sgn = err > 0.0f ? 1.0f : (err < 0.0f ? -1.0f : 0.0f);
            const float dz3 = wt * sgn * yp * (1.0f - yp);
            put(kRowD3, dz3);
            float dz2[9], dz1[12];
#pragma unroll
            for (int o = 0; o < 9; ++o) {
                dz2[o] = h3[o] > 0.0f ? dz3 * th[kP_W3 + o] : 0.0f;
                put(kRowF + o, f[o]);
                put(kRowH1 + o, h1[o]);
                put(kRowH3 + o, h3[o]);
                put(kRowD2 + o, dz2[o]);
            }
#pragma unroll
            for (int i = 0; i < 12; ++i) {
                float d = 0.0f;
#pragma unroll
                for (int o = 0; o < 9; ++o) d = fmaf(th[kP_W2 + 12 * o + i], dz2[o], d);
                dz1[i] = h2[i] > 0.0f ? d : 0.0f;
                put(kRowH2 + i, h2[i]);
                put(kRowD1 + i, dz1[i]);
            }
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                float d = 0.0f;
#pragma unroll
                for (int o = 0; o < 12; ++o) d = fmaf(th[kP_W1 + 9 * o + i], dz1[o], d);
                put(kRowD0 + i, h1[i] > 0.0f ? d : 0.0f);
            }
        }
        __syncthreads();
        if (tid < kTrainSums) {
            float t0 = 0.0f, t1 = 0.0f, t2 = 0.0f, t3 = 0.0f;
#pragma unroll 8
            for (int i = 0; i < kS / 4; ++i) {
                const float4 x = va[i], z = vb[i];
                t0 = fmaf(x.x, z.x, t0);
                t1 = fmaf(x.y, z.y, t1);
                t2 = fmaf(x.z, z.z, t2);
                t3 = fmaf(x.w, z.w, t3);
            }
            sum += (t0 + t1) + (t2 + t3);
        }
        __syncthreads();
    }
    if (tid < kPnetParams) atomicAdd(&a.p.acc[tid], sum);
    else if (tid < kTrainSums) atomicAdd(&a.p.acc_loss[tid - kPnetParams], (double)sum);
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(a.p.ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    // the sums of every block are in acc: Adam (beta 0.9, 0.999) on the mean over the weights
    __threadfence();
    const float wsum = (float)__ldcg(&a.p.acc_loss[1]);
    if (tid < kPnetParams) {
        const float gr = __ldcg(&a.p.acc[tid]) / wsum;
        a.p.grad[tid] = gr;
        const float m = 0.9f * a.p.adam_m[tid] + 0.1f * gr;
        const float v = 0.999f * a.p.adam_v[tid] + 0.001f * gr * gr;
        a.p.adam_m[tid] = m;
        a.p.adam_v[tid] = v;
        const float mh = m / (1.0f - b1t), vh = v / (1.0f - b2t);
        a.p.theta[tid] -= lr * mh / (sqrtf(vh) + 1e-7f);
    } else if (tid < kTrainSums) {
        a.p.loss[tid - kPnetParams] = (float)__ldcg(&a.p.acc_loss[tid - kPnetParams]);
    }
    __syncthreads();
    if (tid < kPnetParams) a.p.acc[tid] = 0.0f;
    else if (tid < kTrainSums) a.p.acc_loss[tid - kPnetParams] = 0.0;
    if (tid == 0) *a.p.ticket = 0u;
}

// Samples per tile: 64, so that a minibatch of 8192 reaches 128 SMs, while
// every block has at most two tiles; beyond that 320 (ten of a block's eleven
// warps in the per-sample pass).
constexpr int kTrainTile = 64, kTrainTileBig = 320;
constexpr size_t train_smem(int s) { return sizeof(float) * kTrainRows * (s + 4); }

int pnet_grid(int64_t rows)
{
    int dev = 0, n_sm = 1;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n_sm < 1) n_sm = 1;
    const int64_t want = (rows + kPnetThreads - 1) / kPnetThreads;
    const int64_t cap = (int64_t)n_sm * 8;
    return (int)(want < 1 ? 1 : (want < cap ? want : cap));
}

}  // namespace

compton_status launch_pnet_infer(compton_ctx* ctx, const float* ux, const float* uy, const float* uz,
                                 const float* kx, const float* ky, const float* kz, int64_t n, float w_e, float w_g,
                                 float p_max, float* r_out, cudaStream_t stream)
{
    if (n <= 0) return COMPTON_OK;
    PnetArgs a{};
    a.p = ctx->pnet;
    a.u[0] = ux;
    a.u[1] = uy;
    a.u[2] = uz;
    a.k[0] = kx;
    a.k[1] = ky;
    a.k[2] = kz;
    a.n = n;
    a.ln_we = logf(w_e);
    a.ln_wg = logf(w_g);
    a.ln_pmax = logf(p_max);
    a.r_out = r_out;
    {
        TimedScope ts_(ctx, COMPTON_K_MLP, stream);
        launch_chained(k_pnet_infer<false>, pnet_grid(n), kPnetThreads, 0, stream, a);
    }
    COMPTON_LAUNCH_CHECK(ctx, "k_pnet_infer");
    return COMPTON_OK;
}

compton_status launch_pnet_decide(compton_ctx* ctx, int64_t rows, const MlpDecide& dec, const float* w_e,
                                  const float* w_g, cudaStream_t stream)
{
    PnetArgs a{};
    a.p = ctx->pnet;
    a.cand = ctx->cand;
    a.n_cand = ctx->n_cand;
    a.dt = dec.dt;
    a.gamma64 = dec.gamma64;
    a.ln_w = logf((float)ctx->cfg.w_over_v);
    a.w_e = w_e;
    a.w_g = w_g;
    a.prob_out = dec.prob_out;
    a.flag_out = dec.flag_out;
    a.accepted = ctx->accepted;
    a.n_accepted = ctx->n_accepted;
    a.stats = ctx->stats;
    a.range = ctx->mlp;
    a.range.range_g2max = ctx->pnet.range[0];
    a.range.range_e2min = ctx->pnet.range[1];
    a.range.range_e2max = ctx->pnet.range[2];
    {
        TimedScope ts_(ctx, COMPTON_K_MLP, stream);
        launch_chained(k_pnet_infer<true>, pnet_grid(rows), kPnetThreads, 0, stream, a);
    }
    COMPTON_LAUNCH_CHECK(ctx, "k_pnet_infer<cand>");
    return COMPTON_OK;
}

compton_status launch_pnet_train_step(compton_ctx* ctx, const float* ux, const float* uy, const float* uz,
                                      const float* kx, const float* ky, const float* kz, const float* y,
                                      const float* w, int64_t n, float w_e, float w_g, float p_max, float lr,
                                      cudaStream_t stream)
{
    if (n <= 0) return COMPTON_EINVAL;
    PnetDev& P = ctx->pnet;
    PnetArgs a{};
    a.p = P;
    a.u[0] = ux;
    a.u[1] = uy;
    a.u[2] = uz;
    a.k[0] = kx;
    a.k[1] = ky;
    a.k[2] = kz;
    a.n = n;
    a.ln_we = logf(w_e);
    a.ln_wg = logf(w_g);
    a.ln_pmax = logf(p_max);
    a.y = y;
    a.wts = w;
    const int64_t step = P.step + 1;
    const float b1t = powf(0.9f, (float)step), b2t = powf(0.999f, (float)step);
    const bool big = n > (int64_t)2 * ctx->n_sm * kTrainTile;
    const int tile = big ? kTrainTileBig : kTrainTile;
    const int64_t tiles = (n + tile - 1) / tile;
    const unsigned grid = (unsigned)(tiles < ctx->n_sm ? tiles : ctx->n_sm);
    const int smem = (int)train_smem(tile);
    if (big)
        COMPTON_CUDA_TRY(ctx, cudaFuncSetAttribute(k_pnet_train<kTrainTileBig>,
                                                   cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    // the launch is the whole step: an injected failure comes before it, so that no failed call has updated anything
    if (inject_fault()) return set_injected_error(ctx, "k_pnet_train");
    if (big) launch_chained(k_pnet_train<kTrainTileBig>, grid, kTrainThreads, smem, stream, a, lr, b1t, b2t);
    else launch_chained(k_pnet_train<kTrainTile>, grid, kTrainThreads, smem, stream, a, lr, b1t, b2t);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return set_cuda_error(ctx, e, "k_pnet_train");
    P.step = step;
    return COMPTON_OK;
}

}  // namespace compton
