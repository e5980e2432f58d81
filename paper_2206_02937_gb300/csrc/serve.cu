// serve.cu -- continuous-batching serving of pre-paired Compton batches.
//
// The paper's network object is invoked "for any given batch of inputs"
// (Sec. 2); a PIC code produces such batches from many tiles and time steps.
// This engine admits pair lists of uneven sizes as they arrive, runs them
// together on the GPU and returns each result as soon as it is done:
//
//   compton_submit    validates a request and queues it (host, thread-safe).
//   engine thread     loops: admits queued requests while a block of the
//                     budgeted pool fits them (first fit, in arrival order);
//                     launches the pending tiles (1024 pairs each) of every
//                     admitted request together; when a launch completes,
//                     requests whose tiles are all done are finished and their
//                     blocks freed.  Up to two launches are in flight.  After
//                     a launch that failed nothing more is launched: its
//                     requests and the unfinished others end with the error,
//                     each once nothing of it is in flight.  When the engine
//                     is stopped, a request with tiles launched is finished (its
//                     outputs are partly written), the others are dropped.
//   compton_poll      returns ENOTREADY or the request's result.
//
// A launch is k_serve over its tiles, then, for the surrogate requests' candidates,
// the network with the decision in its epilogue and k_serve_resolve.  The
// kernels read the caller's inputs and write the caller's outputs, so a pair's
// momenta move once in and once out; a request's block of the pool is its share
// of the budget, and is used as staging only where the caller's arrays overlap
// otherwise than output on its own input.  Only candidates (pairs whose uniform
// lies below the bound of every probability) are evaluated, and only they pass
// through the network, all requests' together.  24 requests of 1,155 to 866,000
// pairs, half of them for the BF16 network: 2274 us with a staged copy of every
// array each way and a network pass per request, 414 us so.
//
// Every pair of request r uses Philox counter (pair index within r, step_r)
// under key seed_r, so a request's result does not depend on what it shares
// the GPU with.  No kernel waits on another or on the host: all coordination
// is host-side through events.
#include <sys/prctl.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstddef>
#include <condition_variable>
#include <deque>
#include <map>
#include <mutex>
#include <thread>
#include <unordered_map>
#include <vector>

#include "ctx.hpp"
#include "device_math.cuh"

namespace compton {

constexpr int kServeThreads = 256;
constexpr int kServePairsPerThread = kPairsPerTile / kServeThreads;
constexpr int kServeCandCap = kPairsPerTile + kServeThreads;  // queued candidates: a tile's and a remainder
constexpr int kServeHitCap = 2 * kServeThreads;               // queued collisions: a batch's and a remainder
constexpr int kMaxTilesPerLaunch = 32768;                     // 33.5M pairs
constexpr int kTileRing = 4;
constexpr uint32_t kServeListMin = 1u << 18, kServeListMax = 1u << 21;  // surrogate candidates of a launch
constexpr int kServeRejects = kMaxTilesPerLaunch;

struct ReqDev {
    const float* in_u[3];
    const float* in_k[3];
    float* out_u[3];
    float* out_k[3];
    const float* dens;   // per pair, or nullptr
    float dens_scalar;
    int mode;
    int copy;            // the outputs are not the inputs: every pair is copied
    uint64_t seed, step;
    unsigned long long* scatters;  // collisions, counted on from request to request of a slot
};

struct TileDev {
    int32_t req;
    int32_t count;
    int64_t first;
};

// A launch's device counters and the tiles it could not take (the candidate
// list was full): they are launched again.
struct ServeControl {
    uint32_t n_cand, n_accepted, n_rejected;
    uint32_t n_reserved;  // candidates of all tiles, those turned away too
    uint32_t n_unseen;    // tiles turned away before their candidates were counted
    int32_t rejected[kServeRejects];
};

namespace {

struct CQEntry {
    int32_t req, p;
    float u0, dens;
};

struct SQEntry {
    int32_t req, p;
    float x, F2;
};

// One more collision of request req for every thread that is here: one atomic
// per request and warp.
__device__ __forceinline__ void count_hit(const ReqDev* reqs, int32_t req)
{
    const unsigned peers = __match_any_sync(__activemask(), req);
    if ((int)(threadIdx.x & 31u) == __ffs(peers) - 1)
        atomicAdd(reqs[req].scatters, (unsigned long long)__popc(peers));
}

// The collision of pair p of a request, from its inputs to its outputs.
__device__ __forceinline__ void serve_resolve(const ReqDev& R, int32_t p, float x, float F2, float ux, float uy, float uz,
                                              float kx, float ky, float kz, float c64sq)
{
    const Philox4 rnd = draw(R.seed, R.step, kStreamAngle, (uint32_t)p);
    const Angle ang = kn_sample_angle(x, rnd.r0 >> 8, F2);
    collide_pair(ux, uy, uz, kx, ky, kz, x, ang, u24_closed0(rnd.r1), c64sq);
    R.out_u[0][p] = ux;
    R.out_u[1][p] = uy;
    R.out_u[2][p] = uz;
    R.out_k[0][p] = kx;
    R.out_k[1][p] = ky;
    R.out_k[2][p] = kz;
}

// Words[i] of lane l of each four lanes becomes word l of the quad's lane i.
__device__ __forceinline__ void quad_transpose(uint32_t (&w)[4])
{
    const bool b0 = threadIdx.x & 1u, b1 = threadIdx.x & 2u;
#pragma unroll
    for (int i = 0; i < 4; i += 2) {
        const uint32_t t = __shfl_xor_sync(0xffffffffu, b0 ? w[i] : w[i + 1], 1);
        if (b0) w[i] = t; else w[i + 1] = t;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const uint32_t t = __shfl_xor_sync(0xffffffffu, b1 ? w[i] : w[i + 2], 2);
        if (b1) w[i] = t; else w[i + 2] = t;
    }
}

// One launch over a list of tiles from any mix of requests.  Per tile: the
// pairs are copied to the outputs (coalesced: a thread takes pairs 256 apart,
// the Bernoulli words come to it from its quad's four Philox blocks), the
// candidates of a plain request go to a queue in shared memory that is
// evaluated 256 at a time, and their collisions to a second one; a surrogate
// request's candidates go with their momenta to the launch's list, which the
// network decides.  Per pair the arithmetic is that of the probability kernel
// on explicit pairs (same device functions).
__global__ void __launch_bounds__(kServeThreads, 3)
    k_serve(const ReqDev* __restrict__ reqs, const TileDev* __restrict__ tiles, int n_tiles, float dt, float gamma64,
            float c64sq, DeviceStats* stats, CandPair* __restrict__ cand, uint32_t cand_cap,
            ServeControl* __restrict__ ctl)
{
    __shared__ CQEntry cq[kServeCandCap];
    __shared__ SQEntry sq[kServeHitCap];
    __shared__ int cn, sn, listed, full;
    __shared__ uint32_t list_base;
    const int tid = threadIdx.x;
    if (tid == 0) cn = sn = 0;
    unsigned my_pairs = 0, my_scat = 0;

    auto evaluate = [&](const CQEntry& e) {
        const ReqDev& R = reqs[e.req];
        const Invariants inv = invariants_f32(R.in_u[0][e.p], R.in_u[1][e.p], R.in_u[2][e.p], R.in_k[0][e.p],
                                              R.in_k[1][e.p], R.in_k[2][e.p]);
        float x = inv.x, v = inv.v;
        if (inv.gamma > gamma64)
            invariants_f64(R.in_u[0][e.p], R.in_u[1][e.p], R.in_u[2][e.p], R.in_k[0][e.p], R.in_k[1][e.p],
                           R.in_k[2][e.p], &x, &v);
        const float F2 = kn_F2(x);
        const float sig = 0.375f * F2;
        const float P = inv.eps > 0.0f ? one_minus_exp_neg(e.dens * dt * sig * v) : 0.0f;
        if (e.u0 < P) {
            ++my_scat;
            count_hit(reqs, e.req);
            sq[atomicAdd(&sn, 1)] = SQEntry{e.req, e.p, x, F2};
        }
    };
    auto resolve = [&](const SQEntry& e) {
        const ReqDev& R = reqs[e.req];
        serve_resolve(R, e.p, e.x, e.F2, R.in_u[0][e.p], R.in_u[1][e.p], R.in_u[2][e.p], R.in_k[0][e.p],
                      R.in_k[1][e.p], R.in_k[2][e.p], c64sq);
    };

    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x) {
        const uint32_t reserved = tid == 0 ? __ldcg(&ctl->n_reserved) : 0u;
        const TileDev T = tiles[t];
        const ReqDev& R = reqs[T.req];
        const bool plain = R.mode == COMPTON_MODE_PLAIN;
        // tiles start at multiples of 1024 pairs; this lane draws the block of
        // its quad's pairs of round tid % 4
        uint32_t words[4];
        {
            const Philox4 r = draw(R.seed, R.step, kStreamScatter,
                                   (uint32_t)((T.first + (tid & 3) * kServeThreads + (tid & ~3)) >> 2));
            words[0] = r.r0, words[1] = r.r1, words[2] = r.r2, words[3] = r.r3;
            quad_transpose(words);
        }
        const uint32_t thr0 = cand_threshold(R.dens_scalar, dt);
        float u[4][3], k[4][3], dens[4];
        int slot[4];
        if (tid == 0) {
            listed = 0;
            full = !plain && reserved > cand_cap;
            if (full) {  // no room for any candidate
                ctl->rejected[atomicAdd(&ctl->n_rejected, 1u)] = t;
                atomicAdd(&ctl->n_unseen, 1u);
            }
        }
        __syncthreads();
        if (full) {
            __syncthreads();
            continue;
        }
#pragma unroll
        for (int rr = 0; rr < kServePairsPerThread; ++rr) {
            const int local = rr * kServeThreads + tid;
            slot[rr] = -1;
            if (local >= T.count) continue;
            const int64_t p = T.first + local;
            dens[rr] = R.dens ? R.dens[p] : R.dens_scalar;
            const bool is_cand = (words[rr] >> 8) < (R.dens ? cand_threshold(dens[rr], dt) : thr0);
            if (R.copy || (is_cand && !plain)) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    u[rr][c] = R.in_u[c][p];
                    k[rr][c] = R.in_k[c][p];
                }
            }
            if (R.copy) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    R.out_u[c][p] = u[rr][c];
                    R.out_k[c][p] = k[rr][c];
                }
            }
            if (is_cand) {
                if (plain) cq[atomicAdd(&cn, 1)] = CQEntry{T.req, (int32_t)p, u24_closed0(words[rr]), dens[rr]};
                else slot[rr] = atomicAdd(&listed, 1);
            }
        }
        __syncthreads();  // the copies of this tile come before its collisions' writes
        if (!plain) {
            // room in the list for all of the tile's candidates, or the tile is launched again
            const int want = listed;
            if (tid == 0) {
                // the reservations that fit are the first ones: what they hold has no gaps
                uint32_t at = want > 0 ? atomicAdd(&ctl->n_reserved, (uint32_t)want) : 0u;
                if (at + (uint32_t)want > cand_cap) {
                    at = 0xFFFFFFFFu;
                    ctl->rejected[atomicAdd(&ctl->n_rejected, 1u)] = t;
                } else if (want > 0) {
                    atomicAdd(&ctl->n_cand, (uint32_t)want);
                }
                list_base = at;
            }
            __syncthreads();
            const uint32_t base = list_base;
            if (base != 0xFFFFFFFFu) {
#pragma unroll
                for (int rr = 0; rr < kServePairsPerThread; ++rr) {
                    const int local = rr * kServeThreads + tid;
                    my_pairs += local < T.count;
                    if (slot[rr] < 0) continue;
                    cand[base + (uint32_t)slot[rr]] =
                        CandPair{(int32_t)(T.first + local), T.req, dens[rr], u24_closed0(words[rr]),
                                 (uint32_t)(T.first + local), {u[rr][0], u[rr][1], u[rr][2]},
                                 {k[rr][0], k[rr][1], k[rr][2]}, 0u};
                }
            }
            __syncthreads();
            continue;
        }
#pragma unroll
        for (int rr = 0; rr < kServePairsPerThread; ++rr) my_pairs += rr * kServeThreads + tid < T.count;
        int nc = cn;
        while (nc >= kServeThreads) {
            nc -= kServeThreads;
            evaluate(cq[nc + tid]);
            __syncthreads();
            const int ns = sn;
            if (ns >= kServeThreads) resolve(sq[ns - kServeThreads + tid]);
            __syncthreads();
            if (tid == 0 && ns >= kServeThreads) sn = ns - kServeThreads;
            __syncthreads();
        }
        if (tid == 0) cn = nc;
        __syncthreads();
    }
    __syncthreads();
    if (tid < cn) evaluate(cq[tid]);
    __syncthreads();
    for (int i = tid; i < sn; i += kServeThreads) resolve(sq[i]);
    for (int d = 16; d > 0; d >>= 1) {
        my_pairs += __shfl_xor_sync(0xffffffffu, my_pairs, d);
        my_scat += __shfl_xor_sync(0xffffffffu, my_scat, d);
    }
    if ((tid & 31) == 0 && my_pairs) atomicAdd(&stats->pairs_tested, (unsigned long long)my_pairs);
    if ((tid & 31) == 0 && my_scat) atomicAdd(&stats->scatters, (unsigned long long)my_scat);
}

// The collisions the network decided (counted there): ie is the pair, ig the
// request's slot.
__global__ void __launch_bounds__(256) k_serve_resolve(const ReqDev* __restrict__ reqs, const AcceptedPair* __restrict__ acc,
                                                       const ServeControl* __restrict__ ctl, float gamma64, float c64sq)
{
    const uint32_t n = ctl->n_accepted;
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const AcceptedPair e = acc[i];
        const ReqDev& R = reqs[e.ig];
        float x = e.x;
        if (x < 0.0f) {  // probability came from the network: the collision needs x
            const Invariants inv = invariants_f32(e.u[0], e.u[1], e.u[2], e.k[0], e.k[1], e.k[2]);
            float v = inv.v;
            x = inv.x;
            if (inv.gamma > gamma64) invariants_f64(e.u[0], e.u[1], e.u[2], e.k[0], e.k[1], e.k[2], &x, &v);
        }
        count_hit(reqs, e.ig);
        serve_resolve(R, e.ie, x, kn_F2(x), e.u[0], e.u[1], e.u[2], e.k[0], e.k[1], e.k[2], c64sq);
    }
}

double now_s()
{
    return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

size_t align256(size_t v) { return (v + 255) / 256 * 256; }

}  // namespace

// ---------------------------------------------------------------------------
// Host engine
// ---------------------------------------------------------------------------
struct ServeReq {
    uint64_t ticket = 0;
    compton_request req{};
    int64_t tiles = 0, launched = 0, done_tiles = 0;
    int64_t flying = 0;  // tiles in launches that are not retired
    double share = 0.0;  // candidates among its pairs, roughly
    std::vector<TileDev> again;  // tiles a full candidate list turned away
    int state = 0;  // 0 queued, 1 admitted, 4 done
    size_t off = 0, bytes = 0;
    int dslot = -1;
    double t_submit = 0, t_admit = 0, t_done = 0;
    compton_status status = COMPTON_OK;
    uint64_t scatters = 0;
};

struct Launch {
    cudaEvent_t ev = nullptr;
    int ring = 0;
    compton_status status = COMPTON_OK;      // of every request in it
    compton_status net_status = COMPTON_OK;  // of its surrogate requests
    double known = 0.0, open_pairs = 0.0;    // candidates expected of its scalar densities, surrogate pairs of the others
    std::vector<std::pair<uint64_t, int64_t>> tiles_per_req;  // ticket, tiles in this launch
};

struct ServeEngine {
    compton_ctx* ctx = nullptr;
    int device = 0;
    void* pool = nullptr;
    void* dev = nullptr;   // the lists below on the device
    void* host = nullptr;  // and those on the host, pinned
    size_t pool_bytes = 0;
    std::map<size_t, size_t> free_blocks;  // offset -> size
    size_t in_use = 0, peak_in_use = 0;
    int max_active = 0;
    ReqDev* reqs_dev = nullptr;
    ReqDev* reqs_host = nullptr;        // pinned staging of the table
    int new_lo = 0, new_hi = -1;        // slots filled since the table was last copied
    unsigned long long* counters = nullptr;   // per device slot: collisions since the start
    unsigned long long* scat_host = nullptr;  // pinned copies of the counters, kTileRing x max_active
    std::vector<unsigned long long> scat_base;  // per slot: its counter when its request was admitted
    std::vector<int> free_slots;
    TileDev* tiles_dev = nullptr;
    TileDev* tiles_host = nullptr;      // pinned, kTileRing x kMaxTilesPerLaunch
    CandList list{};                    // surrogate candidates of a launch
    uint32_t list_cap = 0;
    ServeControl* ctl_dev = nullptr;
    ServeControl* ctl_host = nullptr;   // pinned, kTileRing
    int ring = 0;
    cudaStream_t s_compute = nullptr;
    std::mutex mu;
    std::condition_variable cv;
    std::deque<uint64_t> queued;
    std::deque<uint64_t> active;        // admitted, with tiles to launch, in order of admission
    std::unordered_map<uint64_t, ServeReq> reqs;
    std::deque<Launch> inflight;
    uint64_t next_ticket = 1;
    bool stop = false;
    std::thread worker;
    compton_status fatal = COMPTON_OK;
};

namespace {

bool pool_alloc(ServeEngine* E, size_t bytes, size_t* off)
{
    for (auto it = E->free_blocks.begin(); it != E->free_blocks.end(); ++it) {
        if (it->second >= bytes) {
            *off = it->first;
            const size_t rest = it->second - bytes;
            const size_t at = it->first + bytes;
            E->free_blocks.erase(it);
            if (rest) E->free_blocks[at] = rest;
            E->in_use += bytes;
            E->peak_in_use = std::max(E->peak_in_use, E->in_use);
            return true;
        }
    }
    return false;
}

void pool_free(ServeEngine* E, size_t off, size_t bytes)
{
    auto it = E->free_blocks.emplace(off, bytes).first;
    auto next = std::next(it);
    if (next != E->free_blocks.end() && it->first + it->second == next->first) {
        it->second += next->second;
        E->free_blocks.erase(next);
    }
    if (it != E->free_blocks.begin()) {
        auto prev = std::prev(it);
        if (prev->first + prev->second == it->first) {
            prev->second += it->second;
            E->free_blocks.erase(it);
        }
    }
    E->in_use -= bytes;
}

size_t request_bytes(const compton_request& r)
{
    const size_t per_pair = 7 + (r.mode != COMPTON_MODE_PLAIN ? 1 : 0);
    return align256((size_t)r.n * per_pair * sizeof(float)) + 256;
}

// Whether an output of the request shares memory with an input otherwise than
// as that same input (momentum component on itself, from the same address).
bool overlaps_inputs(const compton_request& r)
{
    const char* in[7] = {(const char*)r.ux_in_dev, (const char*)r.uy_in_dev, (const char*)r.uz_in_dev,
                         (const char*)r.kx_in_dev, (const char*)r.ky_in_dev, (const char*)r.kz_in_dev,
                         (const char*)r.n_dens_dev};
    const char* out[6] = {(const char*)r.ux_out_dev, (const char*)r.uy_out_dev, (const char*)r.uz_out_dev,
                          (const char*)r.kx_out_dev, (const char*)r.ky_out_dev, (const char*)r.kz_out_dev};
    const size_t bytes = (size_t)r.n * sizeof(float);
    for (int o = 0; o < 6; ++o)
        for (int i = 0; i < 7; ++i)
            if (in[i] && !(i == o && in[i] == out[o]) && in[i] < out[o] + bytes && out[o] < in[i] + bytes) return true;
    return false;
}

// A CUDA call of the engine: its failure ends the serving.
bool note(ServeEngine* E, cudaError_t e)
{
    if (e == cudaSuccess) return true;
    cudaGetLastError();
    E->fatal = set_cuda_error(E->ctx, e, "serve engine");
    return false;
}

// Admit queued requests in arrival order while blocks fit (a request that
// does not fit waits; later, smaller ones may pass it).
void admit(ServeEngine* E)
{
    for (auto it = E->queued.begin(); it != E->queued.end();) {
        ServeReq& R = E->reqs[*it];
        if (E->free_slots.empty() || E->fatal != COMPTON_OK) break;
        size_t off;
        if (!pool_alloc(E, R.bytes, &off)) {
            ++it;
            continue;
        }
        R.off = off;
        R.dslot = E->free_slots.back();
        E->free_slots.pop_back();
        R.state = 1;
        R.t_admit = now_s();
        const int64_t n = R.req.n;
        const float* src[6] = {R.req.ux_in_dev, R.req.uy_in_dev, R.req.uz_in_dev,
                               R.req.kx_in_dev, R.req.ky_in_dev, R.req.kz_in_dev};
        float* dst[6] = {R.req.ux_out_dev, R.req.uy_out_dev, R.req.uz_out_dev,
                         R.req.kx_out_dev, R.req.ky_out_dev, R.req.kz_out_dev};
        ReqDev d{};
        d.dens = R.req.n_dens_dev;
        if (overlaps_inputs(R.req)) {
            // the outputs would overwrite inputs of other pairs: the inputs are staged in the block
            float* base = reinterpret_cast<float*>(static_cast<char*>(E->pool) + off);
            for (int c = 0; c < 7; ++c) {
                const float* from = c < 6 ? src[c] : R.req.n_dens_dev;
                if (!from) continue;
                note(E, cudaMemcpyAsync(base + (size_t)c * n, from, n * sizeof(float), cudaMemcpyDeviceToDevice,
                                        E->s_compute));
                if (c < 6) src[c] = base + (size_t)c * n;
                else d.dens = base + (size_t)c * n;
            }
        }
        for (int c = 0; c < 3; ++c) {
            d.in_u[c] = src[c];
            d.in_k[c] = src[3 + c];
            d.out_u[c] = dst[c];
            d.out_k[c] = dst[3 + c];
        }
        for (int c = 0; c < 6; ++c) d.copy |= src[c] != dst[c];
        d.dens_scalar = R.req.n_dens;
        d.mode = (int)R.req.mode;
        d.seed = R.req.seed;
        d.step = R.req.step;
        d.scatters = E->counters + R.dslot;
        E->reqs_host[R.dslot] = d;
        E->new_lo = E->new_hi < 0 ? R.dslot : std::min(E->new_lo, R.dslot);
        E->new_hi = std::max(E->new_hi, R.dslot);
        E->active.push_back(R.ticket);
        it = E->queued.erase(it);
    }
}

// The share of a request's pairs that are candidates, roughly (a launch takes no
// more surrogate tiles than its list will hold; what it turns away is launched
// again).  Densities per pair are on the device: a quarter, until the first
// launch of the request has counted them (retire).
double candidate_share(const compton_request& r, double dt)
{
    if (r.n_dens_dev) return 0.25;
    const double share = 1.0 - std::exp(-2.001 * (double)r.n_dens * dt);
    return share < 1.0 ? share : 1.0;
}

// The launch's table, tiles and k_serve.
compton_status launch_serve(ServeEngine* E, const TileDev* th, TileDev* td, int nt)
{
    compton_ctx* ctx = E->ctx;
    const compton_config& cfg = ctx->cfg;
    cudaStream_t s = E->s_compute;
    if (E->new_hi >= 0) {
        COMPTON_CUDA_TRY(ctx, cudaMemcpyAsync(E->reqs_dev + E->new_lo, E->reqs_host + E->new_lo,
                                              sizeof(ReqDev) * (E->new_hi - E->new_lo + 1), cudaMemcpyHostToDevice, s));
        E->new_hi = -1;
    }
    COMPTON_CUDA_TRY(ctx, cudaMemcpyAsync(td, th, nt * sizeof(TileDev), cudaMemcpyHostToDevice, s));
    COMPTON_CUDA_TRY(ctx, cudaMemsetAsync(E->ctl_dev, 0, offsetof(ServeControl, rejected), s));
    const int grid = std::min(nt, ctx->n_sm * 3);
    k_serve<<<grid, kServeThreads, 0, s>>>(E->reqs_dev, td, nt, (float)cfg.dt, cfg.gamma_fp64_threshold,
                                           cfg.collide_fp64_threshold * cfg.collide_fp64_threshold, ctx->stats,
                                           E->list.cand, E->list_cap, E->ctl_dev);
    COMPTON_LAUNCH_CHECK(ctx, "k_serve");
    return COMPTON_OK;
}

// The network, the decisions and the collisions of the launch's candidates,
// about `rows` of them (a full list at most).
compton_status launch_candidates(ServeEngine* E, int mode, int64_t rows)
{
    compton_ctx* ctx = E->ctx;
    const compton_config& cfg = ctx->cfg;
    cudaStream_t s = E->s_compute;
    const MlpDecide dec{(float)cfg.dt, cfg.gamma_fp64_threshold, nullptr, nullptr, false};
    const bool fused = mode != COMPTON_MODE_MLP_FP32;
    compton_status st = launch_mlp_infer(ctx, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, rows,
                                         (compton_mode)mode, E->list.r, s, false, false, fused ? &dec : nullptr,
                                         &E->list);
    if (st == COMPTON_OK && !fused) st = launch_decide(ctx, E->list, rows, s);
    if (st != COMPTON_OK) return st;
    const int rgrid = (int)std::min<int64_t>((rows + 255) / 256, (int64_t)ctx->n_sm * 32);
    k_serve_resolve<<<rgrid, 256, 0, s>>>(E->reqs_dev, E->list.accepted, E->ctl_dev, cfg.gamma_fp64_threshold,
                                          cfg.collide_fp64_threshold * cfg.collide_fp64_threshold);
    COMPTON_LAUNCH_CHECK(ctx, "k_serve_resolve");
    return COMPTON_OK;
}

// The counters and the tiles turned away, to the host, and the launch's event.
compton_status launch_results(ServeEngine* E, Launch& L, int nt)
{
    compton_ctx* ctx = E->ctx;
    cudaStream_t s = E->s_compute;
    COMPTON_CUDA_TRY(ctx, cudaMemcpyAsync(E->ctl_host + L.ring, E->ctl_dev,
                                          offsetof(ServeControl, rejected) + nt * sizeof(int32_t),
                                          cudaMemcpyDeviceToHost, s));
    int hi = 0;
    for (const auto& tr : L.tiles_per_req) hi = std::max(hi, E->reqs[tr.first].dslot);
    COMPTON_CUDA_TRY(ctx, cudaMemcpyAsync(E->scat_host + (size_t)L.ring * E->max_active, E->counters,
                                          sizeof(unsigned long long) * (hi + 1), cudaMemcpyDeviceToHost, s));
    COMPTON_CUDA_TRY(ctx, cudaEventCreateWithFlags(&L.ev, cudaEventDisableTiming));
    COMPTON_CUDA_TRY(ctx, cudaEventRecord(L.ev, s));
    return COMPTON_OK;
}

void launch_tiles(ServeEngine* E)
{
    if (E->active.empty() || E->fatal != COMPTON_OK) return;
    TileDev* th = E->tiles_host + (size_t)E->ring * kMaxTilesPerLaunch;
    TileDev* td = E->tiles_dev + (size_t)E->ring * kMaxTilesPerLaunch;
    int nt = 0;
    Launch L;
    L.ring = E->ring;
    // one network mode per launch: that of the first surrogate request in line
    int mode = COMPTON_MODE_PLAIN;
    double cand = 0.0;
    std::deque<uint64_t> rest;
    for (const uint64_t ticket : E->active) {
        ServeReq& R = E->reqs[ticket];
        const bool surrogate = R.req.mode != COMPTON_MODE_PLAIN;
        if (surrogate && mode == COMPTON_MODE_PLAIN) mode = (int)R.req.mode;
        int64_t take = 0;
        if (!surrogate || mode == (int)R.req.mode) {
            while ((R.launched < R.tiles || !R.again.empty()) && nt < kMaxTilesPerLaunch) {
                if (surrogate) {
                    const double c = R.share * kPairsPerTile;
                    if (cand > 0.0 && cand + c > 0.95 * E->list_cap) break;
                    cand += c;
                    if (R.req.n_dens_dev) L.open_pairs += kPairsPerTile;
                    else L.known += c;
                }
                if (!R.again.empty()) {
                    th[nt++] = R.again.back();
                    R.again.pop_back();
                } else {
                    const int64_t first = R.launched * kPairsPerTile;
                    th[nt++] = TileDev{R.dslot, (int32_t)std::min<int64_t>(kPairsPerTile, R.req.n - first), first};
                    ++R.launched;
                }
                ++take;
            }
        }
        if (take) L.tiles_per_req.emplace_back(ticket, take);
        R.flying += take;
        if (R.launched < R.tiles || !R.again.empty()) rest.push_back(ticket);
    }
    E->active.swap(rest);
    if (nt == 0) return;
    L.status = launch_serve(E, th, td, nt);
    if (L.status == COMPTON_OK && mode != COMPTON_MODE_PLAIN)
        // the grids are sized for the list the host expects, at most a full one
        L.net_status = launch_candidates(E, mode, (int64_t)std::min<double>(E->list_cap, 1.2 * cand + 4096.0));
    if (L.status == COMPTON_OK) L.status = launch_results(E, L, nt);
    if (L.status != COMPTON_OK) {
        // no event to wait for: everything before has to end here
        cudaStreamSynchronize(E->s_compute);
        cudaGetLastError();
        E->fatal = L.status;
    } else if (L.net_status != COMPTON_OK) {
        E->fatal = L.net_status;
    }
    E->inflight.push_back(std::move(L));
    E->ring = (E->ring + 1) % kTileRing;
}

// A request's end: its block and slot are given back, its result is ready.
void finish(ServeEngine* E, ServeReq& R, compton_status status)
{
    R.state = 4;
    R.status = status;
    R.t_done = now_s();
    if (R.dslot >= 0) {
        pool_free(E, R.off, R.bytes);
        E->free_slots.push_back(R.dslot);
        R.dslot = -1;
    } else {
        R.t_admit = R.t_done;
    }
}

void retire(ServeEngine* E)
{
    while (!E->inflight.empty()) {
        Launch& L = E->inflight.front();
        const cudaError_t q = L.ev ? cudaEventQuery(L.ev) : cudaSuccess;
        if (q == cudaErrorNotReady) break;
        if (!note(E, q)) L.status = E->fatal;
        const bool read = L.status == COMPTON_OK;  // the launch's counters are on the host
        ServeControl* ch = E->ctl_host + L.ring;
        const uint32_t n_rejected = read ? ch->n_rejected : 0;
        const TileDev* th = E->tiles_host + (size_t)L.ring * kMaxTilesPerLaunch;
        // candidates among the pairs whose densities are on the device
        double share = 0.0;
        const double seen = L.open_pairs - (read ? (double)ch->n_unseen * kPairsPerTile : 0.0);
        if (read && seen > 0.0) share = std::min(1.0, std::max(1e-3, ((double)ch->n_reserved - L.known) / seen));
        std::unordered_map<int, int64_t> turned_away;  // slot -> tiles
        for (uint32_t i = 0; i < n_rejected; ++i) ++turned_away[th[ch->rejected[i]].req];
        for (auto& tr : L.tiles_per_req) {
            ServeReq& R = E->reqs[tr.first];
            const compton_status st = L.status == COMPTON_OK && R.req.mode != COMPTON_MODE_PLAIN ? L.net_status : L.status;
            if (R.status == COMPTON_OK) R.status = st;
            const auto it = turned_away.find(R.dslot);
            const int64_t away = it == turned_away.end() ? 0 : it->second;
            R.flying -= tr.second;
            if (share > 0.0 && R.req.n_dens_dev) R.share = share;
            R.done_tiles += tr.second - away;
            if (away) {
                if (R.launched == R.tiles && R.again.empty()) E->active.push_back(R.ticket);
                for (uint32_t i = 0; i < n_rejected; ++i)
                    if (th[ch->rejected[i]].req == R.dslot) R.again.push_back(th[ch->rejected[i]]);
            }
            if (R.done_tiles == R.tiles) {
                if (read) {
                    const unsigned long long count = E->scat_host[(size_t)L.ring * E->max_active + R.dslot];
                    R.scatters = count - E->scat_base[R.dslot];
                    E->scat_base[R.dslot] = count;
                }
                finish(E, R, R.status);
            }
        }
        if (L.ev) cudaEventDestroy(L.ev);
        E->inflight.pop_front();
    }
    if (E->fatal == COMPTON_OK) return;
    // nothing more is launched: the other requests end as well, those with
    // tiles in flight when these are retired
    for (const uint64_t ticket : E->queued) finish(E, E->reqs[ticket], E->fatal);
    E->queued.clear();
    std::deque<uint64_t> rest;
    for (const uint64_t ticket : E->active) {
        ServeReq& R = E->reqs[ticket];
        if (R.flying > 0) rest.push_back(ticket);
        else finish(E, R, R.status != COMPTON_OK ? R.status : E->fatal);
    }
    E->active.swap(rest);
}

void engine_loop(ServeEngine* E)
{
    cudaSetDevice(E->device);
    prctl(PR_SET_TIMERSLACK, 1000);  // the 20 us sleeps below: wake within a microsecond of them
    std::unique_lock<std::mutex> lk(E->mu);
    for (;;) {
        retire(E);
        if (E->stop) {
            E->queued.clear();
            std::deque<uint64_t> begun;
            for (const uint64_t ticket : E->active)
                if (E->reqs[ticket].launched > 0) begun.push_back(ticket);
            E->active.swap(begun);
            if (E->inflight.empty() && E->active.empty()) break;
        } else {
            admit(E);
        }
        if (E->inflight.size() < 2) launch_tiles(E);
        const bool busy = !E->inflight.empty() || !E->queued.empty() || !E->active.empty();
        if (busy) {
            lk.unlock();
            std::this_thread::sleep_for(std::chrono::microseconds(20));
            lk.lock();
        } else {
            E->cv.wait_for(lk, std::chrono::milliseconds(5));
        }
    }
}

}  // namespace

void serve_stop_free(ServeEngine* E);

compton_status serve_start(compton_ctx* ctx, uint64_t pool_bytes, int32_t max_active)
{
    if (ctx->serve) return COMPTON_EINVAL;
    auto* E = new (std::nothrow) ServeEngine();
    if (!E) return COMPTON_ENOMEM;
    E->ctx = ctx;
    E->device = ctx->cfg.device;
    E->pool_bytes = pool_bytes;
    E->max_active = max_active;
    // one candidate for two pairs that the pool admits, within the bounds: a
    // launch has fixed costs of about 30 us and a last wave of collisions.  8
    // million pairs of densities 200 (all candidates) for the BF16 network, known
    // to the host / per pair on the device: 4119 and 4361 us with 2^18 and no
    // count of the candidates seen, 3966 and 4060 with the count, 2742 and 2883
    // with 2^21 and no work spent on tiles that find the list full.
    E->list_cap = (uint32_t)std::min<uint64_t>(kServeListMax, std::max<uint64_t>(kServeListMin, pool_bytes / 64));
    cudaError_t e = inject_fault() ? cudaErrorMemoryAllocation : cudaMalloc(&E->pool, pool_bytes);
    // one allocation each for the device's and the host's (pinned) lists
    const size_t slots = (size_t)max_active;
    size_t dev_bytes = 0, host_bytes = 0;
    const auto take = [](size_t& used, size_t bytes) {
        const size_t at = used;
        used += align256(bytes);
        return at;
    };
    const size_t d_cand = take(dev_bytes, sizeof(CandPair) * E->list_cap);
    const size_t d_acc = take(dev_bytes, sizeof(AcceptedPair) * E->list_cap);
    const size_t d_r = take(dev_bytes, sizeof(float) * E->list_cap);
    const size_t d_tiles = take(dev_bytes, sizeof(TileDev) * kMaxTilesPerLaunch * kTileRing);
    const size_t d_reqs = take(dev_bytes, sizeof(ReqDev) * slots);
    const size_t d_counters = take(dev_bytes, sizeof(unsigned long long) * slots);
    const size_t d_ctl = take(dev_bytes, sizeof(ServeControl));
    const size_t h_tiles = take(host_bytes, sizeof(TileDev) * kMaxTilesPerLaunch * kTileRing);
    const size_t h_reqs = take(host_bytes, sizeof(ReqDev) * slots);
    const size_t h_scat = take(host_bytes, sizeof(unsigned long long) * slots * kTileRing);
    const size_t h_ctl = take(host_bytes, sizeof(ServeControl) * kTileRing);
    if (e == cudaSuccess) e = cudaMalloc(&E->dev, dev_bytes);
    if (e == cudaSuccess) e = cudaMallocHost(&E->host, host_bytes);
    if (e == cudaSuccess) {
        char* d = static_cast<char*>(E->dev);
        char* h = static_cast<char*>(E->host);
        E->list.cand = reinterpret_cast<CandPair*>(d + d_cand);
        E->list.accepted = reinterpret_cast<AcceptedPair*>(d + d_acc);
        E->list.r = reinterpret_cast<float*>(d + d_r);
        E->tiles_dev = reinterpret_cast<TileDev*>(d + d_tiles);
        E->reqs_dev = reinterpret_cast<ReqDev*>(d + d_reqs);
        E->counters = reinterpret_cast<unsigned long long*>(d + d_counters);
        E->ctl_dev = reinterpret_cast<ServeControl*>(d + d_ctl);
        E->tiles_host = reinterpret_cast<TileDev*>(h + h_tiles);
        E->reqs_host = reinterpret_cast<ReqDev*>(h + h_reqs);
        E->scat_host = reinterpret_cast<unsigned long long*>(h + h_scat);
        E->ctl_host = reinterpret_cast<ServeControl*>(h + h_ctl);
    }
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&E->s_compute, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaMemsetAsync(E->counters, 0, sizeof(unsigned long long) * slots, E->s_compute);
    if (e != cudaSuccess) {
        cudaGetLastError();
        serve_stop_free(E);
        return COMPTON_ENOMEM;
    }
    E->list.n_cand = &E->ctl_dev->n_cand;
    E->list.n_accepted = &E->ctl_dev->n_accepted;
    E->scat_base.assign(max_active, 0);
    E->free_blocks[0] = pool_bytes;
    for (int i = max_active - 1; i >= 0; --i) E->free_slots.push_back(i);
    ctx->serve = E;
    E->worker = std::thread(engine_loop, E);
    return COMPTON_OK;
}

void serve_stop_free(ServeEngine* E)
{
    if (E->pool) cudaFree(E->pool);
    if (E->dev) cudaFree(E->dev);
    if (E->host) cudaFreeHost(E->host);
    if (E->s_compute) cudaStreamDestroy(E->s_compute);
    for (auto& L : E->inflight)
        if (L.ev) cudaEventDestroy(L.ev);
    delete E;
}

compton_status serve_stop(compton_ctx* ctx)
{
    ServeEngine* E = ctx->serve;
    if (!E) return COMPTON_OK;
    {
        std::lock_guard<std::mutex> lk(E->mu);
        E->stop = true;
    }
    E->cv.notify_all();
    if (E->worker.joinable()) E->worker.join();
    cudaStreamSynchronize(E->s_compute);
    serve_stop_free(E);
    ctx->serve = nullptr;
    return COMPTON_OK;
}

compton_status serve_submit(compton_ctx* ctx, const compton_request* r, uint64_t* ticket)
{
    ServeEngine* E = ctx->serve;
    if (!E) return COMPTON_EINVAL;
    const size_t bytes = request_bytes(*r);
    if (bytes > E->pool_bytes) return COMPTON_ERANGE;
    std::lock_guard<std::mutex> lk(E->mu);
    if (E->fatal != COMPTON_OK) return E->fatal;
    if (E->queued.size() >= 65536) return COMPTON_EBUSY;
    ServeReq R;
    R.ticket = E->next_ticket++;
    R.req = *r;
    R.tiles = (r->n + kPairsPerTile - 1) / kPairsPerTile;
    R.bytes = bytes;
    R.share = candidate_share(*r, ctx->cfg.dt);
    R.t_submit = now_s();
    *ticket = R.ticket;
    E->reqs.emplace(R.ticket, R);
    E->queued.push_back(R.ticket);
    E->cv.notify_all();
    return COMPTON_OK;
}

compton_status serve_poll(compton_ctx* ctx, uint64_t ticket, compton_result* out)
{
    ServeEngine* E = ctx->serve;
    if (!E) return COMPTON_EINVAL;
    std::lock_guard<std::mutex> lk(E->mu);
    auto it = E->reqs.find(ticket);
    if (it == E->reqs.end()) return COMPTON_EINVAL;
    ServeReq& R = it->second;
    if (R.state != 4) return COMPTON_ENOTREADY;
    const compton_status st = R.status;
    out->status = st;
    out->scatters = R.scatters;
    out->latency_s = R.t_done - R.t_submit;
    out->queue_s = R.t_admit - R.t_submit;
    E->reqs.erase(it);
    return st;
}

compton_status serve_info(compton_ctx* ctx, uint64_t* in_use, uint64_t* peak, uint64_t* pool)
{
    ServeEngine* E = ctx->serve;
    if (!E) return COMPTON_EINVAL;
    std::lock_guard<std::mutex> lk(E->mu);
    *in_use = E->in_use;
    *peak = E->peak_in_use;
    *pool = E->pool_bytes;
    return COMPTON_OK;
}

}  // namespace compton
