// bin_pairs.cu -- binning and random in-cell pairing (arXiv 2206.02937,
// Sec. 3.1, first step: "the simulation space is divided into collision
// cells, in which the particles are binned; from this binning a list of
// colliding leptons and photons is produced for each cell").
//
// Five launches per call (six above 512 scan tiles), both species in each (a
// small call: k_bin_small, which does all before the sort in one, and the sort):
//   k_count        histogram of cell indices by run boundaries, order check
//   k_scan_reduce  per-tile sums of N_e,c, N_g,c and M_c = min(N_e,c, N_g,c)
//   k_scan_blocks  exclusive scan of the tile sums (one CTA; many cells only)
//   k_scan_final   per-cell offsets, CellInfo, tile maps; resets the cursors
//   k_place        input not in cell order only: each particle's index (input
//                  nearly in order) or its record (key, id, momentum) placed
//                  in its cell's segment (arbitrary order inside the segment)
//   k_sort_gather  per-cell sort by (key, id) in shared memory (a bucket
//                  sort of each tile of whole cells), each particle written
//                  to its sorted position
// The order within a cell depends only on (key, id): the atomics of k_place
// decide where a record lands inside its segment, and the sort removes that
// freedom.
#include "ctx.hpp"
#include "device_math.cuh"

namespace compton {
namespace {

constexpr int kSortThreads = 128;
constexpr int kPlaceThreads = 512;   // threads per placement CTA
constexpr int kPlaceCtasPerSm = 16;  // placement CTAs per SM and species
constexpr int kPlaceAloneCells = 4096;  // cells from which records are placed one atomic each (with a search for
                                        // peers in the warp, 301 x 257 cells of 40 + 40 in no order: 361 against
                                        // 348 us for the step; with few cells one address would serialise them)
constexpr int kPlaceUnroll = 4;      // particles whose indices a thread places at once
constexpr int kCountThreads = 1024;  // threads per histogram CTA (256, 512: 1 us slower)

__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }

// ---------------------------------------------------------------------------
// Histogram and order check.  A warp walks one stretch of the positions, 128 at
// a time, four per lane by one vector load; a run of equal cell indices begins
// at the first of the 128 and wherever the index changes.  The lane that holds a
// run's beginning adds its length to the cell: the end is the lane's next
// beginning or, by one shuffle, the first one of a later lane.  So a position
// costs its load and one comparison, and a lane repeats the rest for each
// beginning it holds (one turn for most of input in cell order).
// unsorted[s] counts the positions at which the cell index descends, plus one
// per warp that saw an index outside [0, C): only if it is not zero does the
// placement run, and by its size the placement takes its form (sort_source).
// In large input every fourth warp also looks at its last 128 positions:
// unsorted[2 + s] counts the positions (four times a stretch) of those in whose
// stretch neighbours in the input are not neighbours in the cells (scattered).
//
// What bounds it: instruction issue (113 instructions per 128 positions of input
// in cell order; 140 when every position was looked at as first and last of its
// run).  512^2 cells of 64 + 64: 36.0 us so before, 32.5 now (20 us of reads); a
// tenth of them moved 78 and 71; 128^3 cells of 16 + 16 64.3 and 58.5; 301 x 257
// cells of 40 + 40 in no order 49.3 and 49.2 (one atomic per position).
// ---------------------------------------------------------------------------
template <typename Idx>
__device__ __forceinline__ int4 load_cells4(const int32_t* __restrict__ cell, Idx i, Idx n, bool vec)
{
    if (vec && i + 3 < n) return *reinterpret_cast<const int4*>(cell + i);  // 16-byte aligned: i % 4 == 0
    int4 v = make_int4(-1, -1, -1, -1);
    if (i < n) v.x = cell[i];
    if (i + 1 < n) v.y = cell[i + 1];
    if (i + 2 < n) v.z = cell[i + 2];
    if (i + 3 < n) v.w = cell[i + 3];
    return v;
}

// Particles of a species from which the placement looks at scattered: below,
// the input stays in the L2 while the sort gathers from it.
constexpr int64_t kScatterLook = (int64_t)1 << 22;

// Whether most of 128 consecutive positions lie far from their neighbours in the
// cells (v: four per lane): more than max_runs runs of equal cells (a 32-byte
// sector holds eight words), and 64 positions on another cell than such input in cell order, or some
// two dozen ordered runs of it, would have there (one cell per n / C positions).
__device__ __forceinline__ bool scattered(const int4& v, int64_t n, int64_t C, unsigned max_runs)
{
    const unsigned lane = lane_id();
    const int32_t left = __shfl_up_sync(0xffffffffu, v.w, 1), on = __shfl_down_sync(0xffffffffu, v.x, 16);
    const unsigned begins = __reduce_add_sync(0xffffffffu, (unsigned)(lane == 0 || v.x != left) + (v.y != v.x) +
                                                               (v.z != v.y) + (v.w != v.z));
    const uint32_t near = (uint32_t)(24.0f * 64.0f * (float)C / (float)n) + 8u;
    const unsigned far = __ballot_sync(0xffffffffu, lane < 16u && (uint32_t)on - (uint32_t)v.x > near);
    return begins > max_runs && __popc(far) > 8;
}

// Positions in Idx: 32-bit when every position the grid visits fits (the
// launch checks), else 64-bit.
template <typename Idx>
__global__ void __launch_bounds__(kCountThreads, sizeof(Idx) == 4 ? 2 : 1) k_count(const int32_t* __restrict__ cell_e, int64_t n_e,
                                                        const int32_t* __restrict__ cell_g, int64_t n_g, int64_t C,
                                                        int32_t* __restrict__ count_e, int32_t* __restrict__ count_g,
                                                        uint32_t* __restrict__ unsorted, unsigned max_runs,
                                                        DeviceStats* stats)
{
    chain_start();
    const int s = blockIdx.y;
    const int32_t* __restrict__ cell = s == 0 ? cell_e : cell_g;
    const Idx n = (Idx)(s == 0 ? n_e : n_g);
    int32_t* __restrict__ count = s == 0 ? count_e : count_g;
    const unsigned lane = lane_id(), gt_mask = 0xfffffffeu << lane;
    const bool vec = (reinterpret_cast<uintptr_t>(cell) & 15u) == 0;
    // cell indices are int32, so C above 2^31 admits every non-negative one
    const uint32_t C32 = C > 0x80000000ll ? 0x80000000u : (uint32_t)C;
    uint32_t descents = 0;
    bool bad = false;
    // a warp's positions lie one after another, so the cell index before its
    // next 128 is the last of these; their load is in flight meanwhile
    const int64_t n_groups = ((int64_t)n + 127) / 128, warps = (int64_t)gridDim.x * (kCountThreads / 32);
    const int64_t w = (int64_t)blockIdx.x * (kCountThreads / 32) + (threadIdx.x >> 5);
    Idx base = (Idx)(n_groups * w / warps) * 128;
    const Idx stop = (Idx)(n_groups * (w + 1) / warps) * 128;  // (of whole groups)
    // no index descends from the lowest value
    int32_t before = base > 0 && base < stop ? cell[base - 1] : INT32_MIN;
    auto load = [&](Idx at) {
        if (vec && at + 128 <= n) return *reinterpret_cast<const int4*>(cell + at + 4 * (Idx)lane);
        return load_cells4(cell, (Idx)(at + 4 * (Idx)lane), n, vec);
    };
    int4 q = make_int4(-1, -1, -1, -1), v = q;
    const Idx begin = base;
    if (base < stop) q = load(base);
    for (; base < stop; base += 128) {
        v = q;
        if (base + 128 < stop) q = load(base + 128);
        const int32_t left = __shfl_up_sync(0xffffffffu, v.w, 1), prev = lane == 0 ? before : left;
        // the lane's positions at which a run begins
        uint32_t f = (lane == 0 || v.x != prev ? 1u : 0u) | (v.y != v.x ? 2u : 0u) | (v.z != v.y ? 4u : 0u) |
                     (v.w != v.z ? 8u : 0u);
        uint32_t end = 128u;
        if (base + 128 > n) {  // the last positions of the array
            end = (uint32_t)(n - base);
            f &= 4u * lane >= end ? 0u : end - 4u * lane >= 4u ? 15u : (1u << (end - 4u * lane)) - 1u;
        }
        // where the lane's last run ends: the first beginning in a later lane
        const unsigned later = __ballot_sync(0xffffffffu, f != 0u) & gt_mask;
        const uint32_t first = __shfl_sync(0xffffffffu, 4u * lane + (uint32_t)__ffs((int)f) - 1u, __ffs((int)later) - 1);
        const uint32_t stop_at = later ? first : end;
        while (f) {
            const uint32_t j = (uint32_t)__ffs((int)f) - 1u;
            f &= f - 1u;
            const int32_t c = j & 2u ? (j & 1u ? v.w : v.z) : (j & 1u ? v.y : v.x);
            const int32_t from = j & 2u ? (j & 1u ? v.z : v.y) : (j & 1u ? v.x : prev);
            const uint32_t len = (f ? 4u * lane + (uint32_t)__ffs((int)f) - 1u : stop_at) - 4u * lane - j;
            const bool ok = (uint32_t)c < C32;
            bad |= !ok;
            descents += from > c;
            if (ok) atomicAdd(&count[c], (int32_t)len);
        }
        __syncwarp();
        before = __shfl_sync(0xffffffffu, v.w, 31);  // (the last positions are alone partial)
    }
    const bool any_bad = __any_sync(0xffffffffu, bad);
    descents = __reduce_add_sync(0xffffffffu, descents);
    // every fourth warp, for four (where a quarter of the stretch descends the order is settled)
    const bool apart = (int64_t)n > kScatterLook && (w & 3) == 0 && begin < stop && stop <= n &&
                       (int64_t)descents * 4 < (int64_t)(stop - begin) && scattered(v, (int64_t)n, C, max_runs);
    if (lane == 0) {
        if (any_bad) atomicOr(&stats->error_flags, (unsigned long long)kErrCellRange);
        if (descents + any_bad) atomicAdd(&unsorted[s], descents + any_bad);
        if (apart) atomicAdd(&unsorted[2 + s], 4u * (uint32_t)(stop - begin));
    }
}

// Where the sort reads a species from.  In cell order: the input arrays in
// place.  With fewer descents than a quarter of the particles (a plasma after
// a push, where some crossed into a neighbouring cell; a few ordered runs one
// after another) most of a cell's particles are neighbours in the input: the
// placement writes each particle's index (4 bytes) and the sort gathers
// through it.  Above that (particles in no order: half the positions descend)
// a gather would fetch a 32-byte sector per word, and whole records are placed;
// so too where few positions descend but most are scattered (cell i mod C for
// particle i; short runs of equal cells in no order).
// 512^2 cells, 64 + 64 per cell, a tenth of them moved: the placement takes
// 0.087 ms by index and 0.368 ms by record, the sort after it 0.34 ms each.  The
// same cells with particle i in cell i mod C: 0.278 and 0.784 by index, 0.523 and 0.322 by
// record; runs of three in no order 0.224 and 0.916 against 0.498 and 0.338.
enum SortSource : int { kInPlace = 0, kByIndex = 1, kRecords = 2 };
constexpr uint32_t kIndexPlaced = 0xFFFFFFFFu;  // k_bin_small has placed indices, whatever the order
__device__ __forceinline__ SortSource sort_source(const uint32_t* __restrict__ unsorted, int s, int64_t n)
{
    const uint32_t descents = unsorted[s], apart = unsorted[2 + s];
    if (descents == 0) return kInPlace;
    if (descents == kIndexPlaced) return kByIndex;
    return (int64_t)descents * 4 < n && (int64_t)apart * 2 < n ? kByIndex : kRecords;
}

// ---------------------------------------------------------------------------
// Scan over cells, in three passes.  Values per cell: N_e, N_g, M = min.
// ---------------------------------------------------------------------------
// Sums fit 32 bits: a species has fewer than 2^31 particles.
struct Tri {
    int32_t e, g, m;
};

__device__ __forceinline__ Tri tri_add(Tri a, Tri b) { return {a.e + b.e, a.g + b.g, a.m + b.m}; }

__device__ __forceinline__ Tri warp_incl_scan(Tri v)
{
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t e = __shfl_up_sync(0xffffffffu, v.e, d);
        const int32_t g = __shfl_up_sync(0xffffffffu, v.g, d);
        const int32_t m = __shfl_up_sync(0xffffffffu, v.m, d);
        if (lane_id() >= (unsigned)d) v = {v.e + e, v.g + g, v.m + m};
    }
    return v;
}

// Exclusive scan of one Tri per thread over a block of 256 threads.
__device__ __forceinline__ Tri block_excl_scan_256(Tri v)
{
    __shared__ Tri warp_tot[8];
    const Tri inc = warp_incl_scan(v);
    const int w = threadIdx.x >> 5;
    if (lane_id() == 31) warp_tot[w] = inc;
    __syncthreads();
    Tri before{0, 0, 0};
#pragma unroll
    for (int t = 0; t < 7; ++t)
        if (t < w) before = tri_add(before, warp_tot[t]);
    return {before.e + inc.e - v.e, before.g + inc.g - v.g, before.m + inc.m - v.m};
}

// Four consecutive counts from c0 (a multiple of 4) on, zeros past the end.
static_assert(kScanPer == 4, "a vector of counts per thread");
__device__ __forceinline__ int4 load_counts(const int32_t* __restrict__ count, int64_t c0, int64_t C)
{
    if (c0 + 3 < C) return *reinterpret_cast<const int4*>(count + c0);
    int4 v = make_int4(0, 0, 0, 0);
    if (c0 < C) v.x = count[c0];
    if (c0 + 1 < C) v.y = count[c0 + 1];
    if (c0 + 2 < C) v.z = count[c0 + 2];
    return v;
}

__global__ void __launch_bounds__(256) k_scan_reduce(const int32_t* __restrict__ count_e,
                                                     const int32_t* __restrict__ count_g, int64_t C,
                                                     int64_t* __restrict__ block_sums, int64_t n_tiles)
{
    chain_start();
    const int64_t c0 = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanPer;
    const int4 a = load_counts(count_e, c0, C), b = load_counts(count_g, c0, C);
    Tri v{a.x + a.y + a.z + a.w, b.x + b.y + b.z + b.w, min(a.x, b.x) + min(a.y, b.y) + min(a.z, b.z) + min(a.w, b.w)};
    __shared__ Tri warp_sum[8];
    v = {__reduce_add_sync(0xffffffffu, v.e), __reduce_add_sync(0xffffffffu, v.g),
         __reduce_add_sync(0xffffffffu, v.m)};
    if (lane_id() == 0) warp_sum[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) v = tri_add(v, warp_sum[w]);
        block_sums[blockIdx.x] = v.e;
        block_sums[n_tiles + blockIdx.x] = v.g;
        block_sums[2 * n_tiles + blockIdx.x] = v.m;
    }
}

// One CTA, 1024 tiles at a time, the three sums in one scan with one barrier
// (2048 tiles: 8.4 us with a scan and three barriers per sum, 4.7 so, and
// the scan of 256^3 cells 195 -> 173; a
// stretch of tiles per thread takes 5.2 us there but 60 us longer at 16384).
__global__ void __launch_bounds__(1024) k_scan_blocks(int64_t* __restrict__ block_sums, int64_t n_tiles,
                                                      int64_t* __restrict__ n_pairs)
{
    chain_start();
    __shared__ Tri warp_tot[2][32];
    const int w = threadIdx.x >> 5;
    auto load = [&](int64_t t) {
        return t < n_tiles ? Tri{(int32_t)block_sums[t], (int32_t)block_sums[n_tiles + t],
                                 (int32_t)block_sums[2 * n_tiles + t]}
                           : Tri{0, 0, 0};
    };
    auto shfl = [](const Tri& v, int lane) {
        return Tri{__shfl_sync(0xffffffffu, v.e, lane), __shfl_sync(0xffffffffu, v.g, lane),
                   __shfl_sync(0xffffffffu, v.m, lane)};
    };
    Tri carry{0, 0, 0}, next = load(threadIdx.x);
    int buf = 0;
    for (int64_t base = 0; base < n_tiles; base += 1024, buf ^= 1) {
        const int64_t t = base + threadIdx.x;
        const Tri v = next;
        next = load(t + 1024);
        const Tri inc = warp_incl_scan(v);
        if (lane_id() == 31) warp_tot[buf][w] = inc;
        __syncthreads();  // (the other buffer's readers are behind the next barrier)
        const Tri all = warp_incl_scan(warp_tot[buf][lane_id()]);  // every warp for itself
        const Tri before = shfl(all, w > 0 ? w - 1 : 0), total = shfl(all, 31);
        if (t < n_tiles) {
            block_sums[t] = carry.e + (w > 0 ? before.e : 0) + inc.e - v.e;
            block_sums[n_tiles + t] = carry.g + (w > 0 ? before.g : 0) + inc.g - v.g;
            block_sums[2 * n_tiles + t] = carry.m + (w > 0 ? before.m : 0) + inc.m - v.m;
        }
        carry = tri_add(carry, total);
    }
    if (threadIdx.x == 0) *n_pairs = carry.m;
}

struct ScanFinalArgs {
    int32_t* count_e;
    int32_t* count_g;
    const int64_t* block_sums;
    int64_t n_tiles;
    int64_t C;
    int64_t n_e, n_g;
    int32_t* off_e;
    int32_t* off_g;
    CellInfo* cinfo;
    int32_t* tile_cell;
    int32_t* stile_e;
    int32_t* stile_g;
    int64_t nb_e, nb_g;  // sort tiles per species
    int64_t* n_pairs;
    double w_over_v;
};

// Sort tiles of a species whose first cell is c+1: every b >= 1 with
// o < b*T <= o+n (the tile boundary lies inside or at the end of cell c).
__device__ __forceinline__ void write_sort_tiles(int32_t* stile, int64_t nb, uint32_t o, uint32_t n, int64_t c)
{
    if (n == 0) return;
    const uint32_t b_lo = o / kSortTile + 1;
    uint32_t b_hi = (o + n) / kSortTile;
    if (b_hi > nb - 1) b_hi = (uint32_t)(nb - 1);
    for (uint32_t b = b_lo; b <= b_hi; ++b) stile[b] = (int32_t)(c + 1);
}

// The maps' entries of cell c, except its offsets: counts ne, ng, exclusive prefixes p, np_total pairs in all.
__device__ __forceinline__ void scan_cell(const ScanFinalArgs& a, int64_t c, int32_t ne, int32_t ng, const Tri& p,
                                          int64_t np_total)
{
    const uint32_t m = (uint32_t)(ne < ng ? ne : ng), end = (uint32_t)p.m + m;
    const int32_t nmax = ne > ng ? ne : ng;
    CellInfo ci;
    ci.pair_off = p.m;
    ci.e_start = p.e;
    ci.g_start = p.g;
    ci.dens = (float)((double)nmax * a.w_over_v);
    a.cinfo[c] = ci;
    if (m > 0) {
        // scatter tiles whose first pair lies in [p.m, p.m + m)
        for (uint32_t t = ((uint32_t)p.m + kPairsPerTile - 1) / kPairsPerTile; t * kPairsPerTile < end; ++t)
            a.tile_cell[t] = (int32_t)c;
        if (end == np_total) a.tile_cell[(np_total + kPairsPerTile - 1) / kPairsPerTile] = (int32_t)c;
    }
    write_sort_tiles(a.stile_e, a.nb_e, (uint32_t)p.e, (uint32_t)ne, c);
    write_sort_tiles(a.stile_g, a.nb_g, (uint32_t)p.g, (uint32_t)ng, c);
    if (c == a.C - 1) {
        a.off_e[a.C] = p.e + ne;
        a.off_g[a.C] = p.g + ng;
    }
}

__device__ __forceinline__ void scan_ends(const ScanFinalArgs& a)
{
    a.stile_e[0] = 0;
    a.stile_g[0] = 0;
    a.stile_e[a.nb_e] = (int32_t)a.C;
    a.stile_g[a.nb_g] = (int32_t)a.C;
}

// The sums of the tiles before this block's, and the pairs of all tiles in
// *total_m: each block adds them up itself, which takes it about as long as
// waiting for one block's scan of them and saves that launch.
__device__ __forceinline__ Tri tiles_before(const ScanFinalArgs& a, int32_t* total_m)
{
    __shared__ int4 warp_sum[8];
    int4 s = make_int4(0, 0, 0, 0);
    for (int64_t t = threadIdx.x; t < a.n_tiles; t += 256) {
        const int32_t m = (int32_t)a.block_sums[2 * a.n_tiles + t];
        s.w += m;
        if (t < (int64_t)blockIdx.x) {
            s.x += (int32_t)a.block_sums[t];
            s.y += (int32_t)a.block_sums[a.n_tiles + t];
            s.z += m;
        }
    }
    s = make_int4(__reduce_add_sync(0xffffffffu, s.x), __reduce_add_sync(0xffffffffu, s.y),
                  __reduce_add_sync(0xffffffffu, s.z), __reduce_add_sync(0xffffffffu, s.w));
    if (lane_id() == 0) warp_sum[threadIdx.x >> 5] = s;
    __syncthreads();
    Tri sum{0, 0, 0};
    int32_t tm = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        const int4 t = warp_sum[w];
        sum = tri_add(sum, Tri{t.x, t.y, t.z});
        tm += t.w;
    }
    *total_m = tm;
    return sum;
}

// What bounds it: the stores of the maps (24 bytes per cell and the cleared
// counts' 8) and, with few tiles, its chain of loads and barriers.  2 million
// cells: 31 us with 64-bit sums and a load and a store per count, 21 us so.
// kOwnPrefix: block_sums hold the tiles' sums (k_scan_blocks has not run).
template <bool kOwnPrefix>
__global__ void __launch_bounds__(256) k_scan_final(const __grid_constant__ ScanFinalArgs a)
{
    chain_start();
    const int64_t c0 = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanPer;
    const int4 ce = load_counts(a.count_e, c0, a.C), cg = load_counts(a.count_g, c0, a.C);
    const int32_t ne[kScanPer] = {ce.x, ce.y, ce.z, ce.w}, ng[kScanPer] = {cg.x, cg.y, cg.z, cg.w};
    Tri v{0, 0, 0};
#pragma unroll
    for (int j = 0; j < kScanPer; ++j) v = tri_add(v, Tri{ne[j], ng[j], min(ne[j], ng[j])});
    Tri p = block_excl_scan_256(v);
    int32_t np_total;
    if (kOwnPrefix) {
        p = tri_add(p, tiles_before(a, &np_total));
        if (blockIdx.x == 0 && threadIdx.x == 0) *a.n_pairs = np_total;
    } else {
        p = tri_add(p, Tri{(int32_t)a.block_sums[blockIdx.x], (int32_t)a.block_sums[a.n_tiles + blockIdx.x],
                           (int32_t)a.block_sums[2 * a.n_tiles + blockIdx.x]});
        np_total = (int32_t)*a.n_pairs;
    }
    // offsets out; the counts become the insertion cursors of k_place
    if (c0 + 3 < a.C) {
        *reinterpret_cast<int4*>(a.off_e + c0) = make_int4(p.e, p.e + ce.x, p.e + ce.x + ce.y, p.e + ce.x + ce.y + ce.z);
        *reinterpret_cast<int4*>(a.off_g + c0) = make_int4(p.g, p.g + cg.x, p.g + cg.x + cg.y, p.g + cg.x + cg.y + cg.z);
        *reinterpret_cast<int4*>(a.count_e + c0) = make_int4(0, 0, 0, 0);
        *reinterpret_cast<int4*>(a.count_g + c0) = make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int j = 0; j < kScanPer; ++j) {
        const int64_t c = c0 + j;
        if (c >= a.C) break;
        if (c0 + 3 >= a.C) {
            a.off_e[c] = p.e;
            a.off_g[c] = p.g;
            a.count_e[c] = 0;
            a.count_g[c] = 0;
        }
        scan_cell(a, c, ne[j], ng[j], p, np_total);
        p = tri_add(p, Tri{ne[j], ng[j], min(ne[j], ng[j])});
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) scan_ends(a);
}

// ---------------------------------------------------------------------------
// The binning before the sort of a small call, in one launch and one CTA:
// histogram (by run boundaries, as k_count) and order check, the scan over
// cells with all its maps, and, for input not in cell order, the placed
// indices.  The five launches and the memset it replaces take 2 to 5 us each
// however little they do; one CTA walks 8192 + 8192 particles in about as long.
// Whole plain step, its launches in a graph, in order / in no order: 64 cells of
// 64 + 64 20.8 / 26.3 us against 28.8 / 33.7; 128 cells 22.8 / 33.3 against 30.2
// / 36.9; 256 cells (not taken) 25.9 / 44.7 against 31.0 / 38.4.
// ---------------------------------------------------------------------------
constexpr int kSmallThreads = 1024;
constexpr int kSmallCells = 4096;
constexpr int64_t kSmallParticles = 16384;

struct BinSmallArgs {
    const int32_t* cell[2];
    ScanFinalArgs scan;  // n_e, n_g, C, offsets, CellInfo, tile maps
    int64_t* n_pairs;
    int32_t* idx[2];
    uint32_t* unsorted;
    DeviceStats* stats;
};

__global__ void __launch_bounds__(kSmallThreads) k_bin_small(const __grid_constant__ BinSmallArgs a)
{
    chain_start();
    __shared__ int32_t count[2][kSmallCells];  // counts, then the next place of each cell
    __shared__ int3 warp_tot[kSmallThreads / 32];
    __shared__ int disorder[2];
    const int tid = threadIdx.x, C = (int)a.scan.C;
    for (int c = tid; c < C; c += kSmallThreads) count[0][c] = count[1][c] = 0;
    if (tid < 2) disorder[tid] = 0;
    __syncthreads();
    // ---- histogram: half the CTA per species, four consecutive positions per
    // thread, the next four's loads in flight ----
    const int hs = tid / (kSmallThreads / 2), ht = tid % (kSmallThreads / 2);
    bool any_bad = false, dis = false;
    {
        const int32_t* __restrict__ cell = a.cell[hs];
        const int n = (int)(hs == 0 ? a.scan.n_e : a.scan.n_g);
        const bool vec = (reinterpret_cast<uintptr_t>(cell) & 15u) == 0;
        constexpr int kStep = 4 * (kSmallThreads / 2);
        const unsigned lane = lane_id();
        auto edge = [&](int j0) -> int32_t {
            if (lane == 0) return j0 > 0 && j0 - 1 < n ? cell[j0 - 1] : -1;
            if (lane == 31) return j0 + 4 < n ? cell[j0 + 4] : -1;
            return -1;
        };
        int i0 = 4 * ht;
        int4 q = load_cells4(cell, i0, n, vec);
        int32_t e = edge(i0);
        for (int b = 0; b < n; b += kStep, i0 += kStep) {  // the same trips in every thread of the half
            int4 qn = make_int4(-1, -1, -1, -1);
            int32_t en = -1;
            if (b + kStep < n) {
                qn = load_cells4(cell, i0 + kStep, n, vec);
                en = edge(i0 + kStep);
            }
            const int32_t v[4] = {q.x, q.y, q.z, q.w};
            int32_t prev = __shfl_up_sync(0xffffffffu, v[3], 1), next = __shfl_down_sync(0xffffffffu, v[0], 1);
            if (lane == 0) prev = e;
            if (lane == 31) next = e;
            q = qn;
            e = en;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int i = i0 + j;
                if (i >= n) break;
                const int32_t c = v[j], pc = j == 0 ? prev : v[j - 1], nc = j == 3 ? next : v[j + 1];
                const bool ok = (uint32_t)c < (uint32_t)C;
                any_bad |= !ok;
                dis |= !ok || (i > 0 && pc > c);
                const bool first = i == 0 || pc != c, last = i + 1 == n || nc != c;
                if (ok && (first || last)) atomicAdd(&count[hs][c], (last ? i + 1 : 0) - (first ? i : 0));
            }
        }
    }
    if (dis) disorder[hs] = 1;
    if (any_bad) atomicOr(&a.stats->error_flags, (unsigned long long)kErrCellRange);
    __syncthreads();
    // ---- scan over cells, kPer consecutive ones per thread ----
    constexpr int kPer = kSmallCells / kSmallThreads;
    const int c0 = tid * kPer;
    int ne[kPer], ng[kPer];
    int3 v = make_int3(0, 0, 0);  // electrons, photons, pairs
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        ne[j] = c0 + j < C ? count[0][c0 + j] : 0;
        ng[j] = c0 + j < C ? count[1][c0 + j] : 0;
        v = make_int3(v.x + ne[j], v.y + ng[j], v.z + (ne[j] < ng[j] ? ne[j] : ng[j]));
    }
    int3 inc = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, inc.x, d), y = __shfl_up_sync(0xffffffffu, inc.y, d),
                  z = __shfl_up_sync(0xffffffffu, inc.z, d);
        if (lane_id() >= (unsigned)d) inc = make_int3(inc.x + x, inc.y + y, inc.z + z);
    }
    if (lane_id() == 31) warp_tot[tid >> 5] = inc;
    __syncthreads();
    int3 p = make_int3(inc.x - v.x, inc.y - v.y, inc.z - v.z);
    int np_total = 0;
    for (int w = 0; w < kSmallThreads / 32; ++w) {
        const int3 t = warp_tot[w];
        if (w < (tid >> 5)) p = make_int3(p.x + t.x, p.y + t.y, p.z + t.z);
        np_total += t.z;
    }
    const ScanFinalArgs& f = a.scan;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int c = c0 + j;
        if (c >= C) break;
        const Tri t{p.x, p.y, p.z};
        f.off_e[c] = t.e;
        f.off_g[c] = t.g;
        scan_cell(f, c, ne[j], ng[j], t, np_total);
        count[0][c] = p.x;
        count[1][c] = p.y;
        p = make_int3(p.x + ne[j], p.y + ng[j], p.z + (ne[j] < ng[j] ? ne[j] : ng[j]));
    }
    if (tid == 0) {
        scan_ends(f);
        *a.n_pairs = np_total;
    }
    if (tid < 2) a.unsorted[tid] = disorder[tid] ? kIndexPlaced : 0u;
    __syncthreads();
    // ---- places ----
    if (disorder[hs]) {
        const int n = (int)(hs == 0 ? a.scan.n_e : a.scan.n_g);
        const int32_t* __restrict__ cell = a.cell[hs];
        int32_t* __restrict__ idx = a.idx[hs];
        constexpr int kStride = kSmallThreads / 2;
        for (int i = ht; i < n; i += 8 * kStride) {
            int32_t c[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) c[k] = i + k * kStride < n ? cell[i + k * kStride] : -1;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                if ((uint32_t)c[k] < (uint32_t)C) idx[atomicAdd(&count[hs][c[k]], 1)] = i + k * kStride;
        }
    }
}

// ---------------------------------------------------------------------------
// Placement of input not in cell order: each particle takes the next place of
// its cell's segment (off[c] + cursor), where its index or its record (Philox
// key, id, momentum, weight if any) is written.  A record fills one aligned
// 32-byte sector, written as two 16-byte stores, so the scattered writes never
// leave partly written sectors behind.  Input already in cell order skips
// this kernel.  The kernel is bound by the latency of each particle's chain
// (cell index, cursor atomic, write).
// ---------------------------------------------------------------------------
struct PlaceArgs {
    const int32_t* cell[2];
    const uint32_t* id[2];
    const float* u[2][3];
    const float* w[2];  // per-particle weights, or nullptr
    int64_t n[2];
    const int32_t* off[2];
    int32_t* cursor[2];
    const uint32_t* unsorted;
    SortRec* rec[2];  // records, or (kByIndex) the indices as int32
    int64_t C;
    KeyDraw draw;
};

__device__ __forceinline__ void store_rec(SortRec* r, uint32_t key, uint32_t pid, float ux, float uy, float uz,
                                          float w)
{
    uint4* q = reinterpret_cast<uint4*>(r);
    q[0] = make_uint4(key, pid, __float_as_uint(ux), __float_as_uint(uy));
    q[1] = make_uint4(__float_as_uint(uz), __float_as_uint(w), 0u, 0u);
}

// The weight a record carries (its first padding word).
__device__ __forceinline__ float rec_weight(const SortRec* r) { return __uint_as_float(r->pad[0]); }

// The next places of the cells of the warp's 32 particles, one cursor atomic
// per distinct cell: the group's first place in its leader, and this lane's
// leader and rank in its group.
__device__ __forceinline__ void claim_places(const int32_t* __restrict__ off, int32_t* __restrict__ cursor, int c,
                                             int& first_place, int& leader, int& rank)
{
    const unsigned lane = lane_id();
    const unsigned peers = __match_any_sync(0xffffffffu, c);
    leader = __ffs(peers) - 1;
    rank = __popc(peers & ((1u << lane) - 1u));
    first_place = 0;
    if (c >= 0 && lane == (unsigned)leader) first_place = off[c] + atomicAdd(&cursor[c], __popc(peers));
}

template <bool kChained>
__global__ void __launch_bounds__(kPlaceThreads, 2048 / kPlaceThreads) k_place(const __grid_constant__ PlaceArgs a)
{
    if (kChained) chain_start();
    const int s = blockIdx.y;
    const int64_t n = a.n[s];
    const SortSource source = sort_source(a.unsorted, s, n);
    if (source == kInPlace) return;
    const int32_t* __restrict__ cell = a.cell[s];
    const int32_t* __restrict__ off = a.off[s];
    int32_t* __restrict__ cursor = a.cursor[s];
    const unsigned lane = lane_id();
    const int64_t warp = (int64_t)blockIdx.x * (kPlaceThreads / 32) + (threadIdx.x >> 5);
    const int64_t n_warps = (int64_t)gridDim.x * (kPlaceThreads / 32);
    auto load_cell = [&](int64_t i) {
        const int32_t ci = i < n ? cell[i] : -1;
        return ci >= 0 && (int64_t)ci < a.C ? ci : -1;
    };
    if (source == kByIndex) {
        // a warp takes runs of kPlaceUnroll * 32 consecutive particles, their
        // chains (cell, cursor atomic, index) in flight together
        int32_t* __restrict__ idx = reinterpret_cast<int32_t*>(a.rec[s]);
        constexpr int kRun = 32 * kPlaceUnroll;
        for (int64_t r0 = warp * kRun; r0 < n; r0 += n_warps * kRun) {
            int c[kPlaceUnroll], place[kPlaceUnroll], rank[kPlaceUnroll], leader[kPlaceUnroll];
#pragma unroll
            for (int k = 0; k < kPlaceUnroll; ++k) c[k] = load_cell(r0 + 32 * k + lane);
#pragma unroll
            for (int k = 0; k < kPlaceUnroll; ++k) claim_places(off, cursor, c[k], place[k], leader[k], rank[k]);
#pragma unroll
            for (int k = 0; k < kPlaceUnroll; ++k) {
                const int base = __shfl_sync(0xffffffffu, place[k], leader[k]);
                if (c[k] >= 0) idx[(int64_t)base + rank[k]] = (int32_t)(r0 + 32 * k + lane);
            }
        }
        return;
    }
    // whole records.  Particles in no order among many cells seldom share one
    // within a warp: each takes its own place, with no search for peers (scattered
    // input with few descents may hold short runs of equal cells)
    const uint32_t* __restrict__ id = a.id[s];
    const float* __restrict__ wt = a.w[s];
    SortRec* __restrict__ rec = a.rec[s];
    const bool alone = a.C >= kPlaceAloneCells && (int64_t)a.unsorted[s] * 4 >= n;
    for (int64_t r0 = warp * 32; r0 < n; r0 += n_warps * 32) {
        const int64_t i = r0 + lane;
        const int c = load_cell(i);
        int64_t slot = 0;
        if (alone) {
            if (c >= 0) slot = (int64_t)off[c] + atomicAdd(&cursor[c], 1);
        } else {
            int place, leader, rank;
            claim_places(off, cursor, c, place, leader, rank);
            slot = (int64_t)__shfl_sync(0xffffffffu, place, leader) + rank;
        }
        if (c >= 0) {
            const uint32_t pid = id[i];
            const float u0 = a.u[s][0][i], u1 = a.u[s][1][i], u2 = a.u[s][2][i], w = wt ? wt[i] : 0.0f;
            store_rec(rec + slot, a.draw.word0(s, pid), pid, u0, u1, u2, w);
        }
    }
}

// ---------------------------------------------------------------------------
// Per-cell sort by (key, id) and copy into sorted order.
//
// Keys are uniform 32-bit Philox words, so within a cell of n particles the
// bucket floor(key * n / 2^32) is monotone in the key and holds about one
// particle.  A sort tile (whole cells, at most kSortCap particles) gives cell
// c the buckets [a_c, a_c + n_c) at its own positions in the tile, so one
// counting sort over all buckets of the tile sorts every cell at once: a
// histogram in shared memory, one block-wide exclusive scan (its value at the
// start of a cell's buckets is a_c), placement by bucket, and an exact rank
// by (key, id) inside each bucket, after which each element is written to its
// sorted position (entries of neighbouring threads lie in neighbouring
// buckets, so a warp's writes stay within a few sectors).  O(1) work per
// particle, every lane busy whatever the cell sizes.
// ---------------------------------------------------------------------------
struct SortGatherArgs {
    const float* in_u[2][3];
    const uint32_t* in_id[2];
    const float* in_w[2];  // per-particle weights, or nullptr
    float* out_w[2];
    float* out_u[2][3];
    int32_t* out_cell[2];
    uint32_t* out_id[2];
    SortRec* rec[2];  // placed records, or (kByIndex) indices
    const int32_t* off[2];
    const int32_t* stile[2];
    const uint32_t* unsorted;
    int64_t n[2];
    int64_t nb_e;
    KeyDraw draw;
};

// Where a species' particles are read from: the placed records, or the input
// arrays (in place or through the placed indices), with keys drawn from the ids.
struct SortSrc {
    const SortRec* rec;  // kRecords, else nullptr
    const int32_t* idx;  // kByIndex, else nullptr
    const uint32_t* id;
    const float* u[3];
    const float* w;      // weights, or nullptr

    // the input index of position p (no records)
    __device__ __forceinline__ int64_t input(int64_t p) const { return idx ? (int64_t)idx[p] : p; }
};

// The order inside a cell is by (key, id), with the tile slot breaking ties
// between equal ids (invalid input), so the order is total and every sort
// yields a permutation.

__device__ __forceinline__ int bucket_of(uint32_t key, int n) { return (int)__umulhi(key, (uint32_t)n); }

__device__ __forceinline__ void cp_async4(void* smem_dst, const void* gmem_src)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(gmem_src) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

struct SortSmem {
    uint32_t* id;     // [cap] particle id of each tile slot
    int32_t* cnt;     // [kBucketsPerSlot * cap] bucket counts, then starts, then ends
    uint32_t* cmap;   // [cap] a_c | n_c << 16 of the slot's cell; after the
                      // histogram, the keys in bucket order
    uint16_t* ptmp;   // [cap] tile slots grouped by bucket
    uint16_t* pbk;    // [cap] their buckets
    float* us[3];     // [cap] momenta staged from global memory
};

// Placed record gi to tile slot i: momentum and id into shared memory; the
// key is returned.
__device__ __forceinline__ uint32_t fetch_rec(const SortSrc& t, const SortSmem& m, int64_t gi, int i)
{
    const uint4* q = reinterpret_cast<const uint4*>(t.rec + gi);
    const uint4 r0 = q[0], r1 = q[1];
    m.us[0][i] = __uint_as_float(r0.z);
    m.us[1][i] = __uint_as_float(r0.w);
    m.us[2][i] = __uint_as_float(r1.x);
    m.id[i] = r0.y;
    return r0.x;
}

// Buckets per tile slot: a cell of n particles takes kBucketsPerSlot * n
// buckets, so a bucket holds Poisson(1 / kBucketsPerSlot) particles.
constexpr int kBucketsPerSlot = 1;

// Block-wide exclusive scan of cnt[0 .. R) in place (R <= kBucketsPerSlot *
// kSortCap).
__device__ __forceinline__ void block_scan_counts(int32_t* cnt, int R)
{
    constexpr int kPer = (kBucketsPerSlot * kSortCap + kSortThreads - 1) / kSortThreads;
    __shared__ int32_t warp_tot[kSortThreads / 32];
    const int tid = threadIdx.x, lane = (int)lane_id(), w = tid >> 5;
    const int b0 = tid * kPer;
    int v[kPer];
    int sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        v[k] = b0 + k < R ? cnt[b0 + k] : 0;
        sum += v[k];
    }
    int inc = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, inc, d);
        if (lane >= d) inc += o;
    }
    if (lane == 31) warp_tot[w] = inc;
    __syncthreads();
    if (w == 0) {
        int t = lane < kSortThreads / 32 ? warp_tot[lane] : 0;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, t, d);
            if (lane >= d) t += o;
        }
        if (lane < kSortThreads / 32) warp_tot[lane] = t;
    }
    __syncthreads();
    int run = (w > 0 ? warp_tot[w - 1] : 0) + inc - sum;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        if (b0 + k < R) cnt[b0 + k] = run;
        run += v[k];
    }
}

// Sort the tile of cells [c0, c1) (positions o0 .. o0 + R of species s) with
// the whole block.
__device__ __forceinline__ void sort_tile_block(const SortGatherArgs& g, int s, const SortSrc& t, const SortSmem& m,
                                                int64_t c0, int64_t c1, int64_t o0, int R)
{
    const int tid = threadIdx.x;
    const int32_t* __restrict__ off = g.off[s];
    constexpr int kPer = (kSortCap + kSortThreads - 1) / kSortThreads;
    uint32_t key[kPer], pid[kPer];
    // from the input arrays: issue the tile's loads first, so they are in
    // flight while the cell map is built
    if (!t.rec) {
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int i = tid + k * kSortThreads;
            if (i < R) {
                const int64_t q = t.input(o0 + i);
                cp_async4(&m.us[0][i], t.u[0] + q);
                cp_async4(&m.us[1][i], t.u[1] + q);
                cp_async4(&m.us[2][i], t.u[2] + q);
                pid[k] = t.id[q];
            }
        }
    }
    // the tile's cell offsets, staged once (in the placement buffers, unused
    // until later) when they fit; the bucket counters cleared
    const int n_cells = (int)(c1 - c0);
    int32_t* offs = reinterpret_cast<int32_t*>(m.ptmp);
    const bool staged = n_cells < kSortCap;
    if (staged)
        for (int i = tid; i <= n_cells; i += kSortThreads) offs[i] = off[c0 + i] - (int32_t)o0;
    for (int i = tid; i < kBucketsPerSlot * R; i += kSortThreads) m.cnt[i] = 0;
    __syncthreads();
    // cell of every position and the output cell indices: a group of lanes per
    // cell, 32, or 16 or 8 where the tile's cells hold that few on average
    const int gs = R > 16 * n_cells ? 5 : (R > 8 * n_cells ? 4 : 3);
    for (int ci = tid >> gs; ci < n_cells; ci += kSortThreads >> gs) {
        const int a = staged ? offs[ci] : off[c0 + ci] - (int32_t)o0;
        const int n = (staged ? offs[ci + 1] : off[c0 + ci + 1] - (int32_t)o0) - a;
        for (int j = tid & ((1 << gs) - 1); j < n; j += 1 << gs) {
            m.cmap[a + j] = (uint32_t)a | ((uint32_t)n << 16);
            g.out_cell[s][o0 + a + j] = (int32_t)(c0 + ci);
        }
    }
    // keys (and, from placed records, momenta)
    if (t.rec) {
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int i = tid + k * kSortThreads;
            if (i < R) key[k] = fetch_rec(t, m, o0 + i, i);
        }
    } else {
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int i = tid + k * kSortThreads;
            if (i < R) {
                key[k] = g.draw.word0(s, pid[k]);
                m.id[i] = pid[k];
            }
        }
    }
    __syncthreads();
    // bucket histogram; the slots' buckets stay in registers, two 16-bit
    // buckets to a register
    uint32_t bk2[(kPer + 1) / 2];
#pragma unroll
    for (int k = 0; k < (kPer + 1) / 2; ++k) bk2[k] = 0u;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int i = tid + k * kSortThreads;
        if (i < R) {
            const uint32_t cm = m.cmap[i];
            const uint32_t b = kBucketsPerSlot * (cm & 0xffffu) +
                               (uint32_t)bucket_of(key[k], kBucketsPerSlot * (int)(cm >> 16));
            bk2[k >> 1] |= b << ((k & 1) * 16);
            atomicAdd(&m.cnt[b], 1);
        }
    }
    __syncthreads();
    block_scan_counts(m.cnt, kBucketsPerSlot * R);
    __syncthreads();
    // slots, keys and buckets grouped by bucket (the cell map is no longer
    // needed); afterwards cnt[b] = end of bucket b
    uint32_t* pkey = m.cmap;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int i = tid + k * kSortThreads;
        if (i < R) {
            const uint32_t b = (bk2[k >> 1] >> ((k & 1) * 16)) & 0xffffu;
            const int pos = atomicAdd(&m.cnt[b], 1);
            m.ptmp[pos] = (uint16_t)i;
            m.pbk[pos] = (uint16_t)b;
            pkey[pos] = key[k];
        }
    }
    cp_async_wait_all();
    __syncthreads();
    // exact rank inside each bucket, one thread per entry of the grouped list
    // (the end of bucket b - 1 is the start of bucket b, also across cells):
    // neighbouring threads read the same or neighbouring buckets, so a
    // bucket's keys reach them by broadcast; only a key that occurs twice
    // needs the ids (and, for equal ids, the slots) to break the tie
    for (int q = tid; q < R; q += kSortThreads) {
        const int b = m.pbk[q];
        const int lo = b == 0 ? 0 : m.cnt[b - 1];
        const int hi = m.cnt[b];
        const int i = m.ptmp[q];
        int fin = lo;
        if (hi - lo > 1) {
            const uint32_t ki = pkey[q];
            int less = 0, eq = 0;
            if (hi - lo <= 4) {
                // buckets hold Poisson(1) keys: up to four, a fixed unrolled
                // pass (no loop control, the same instructions in every lane)
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    if (lo + r < hi) {
                        const uint32_t kr = pkey[lo + r];
                        less += kr < ki;
                        eq += kr == ki;
                    }
                }
            } else {
                for (int r = lo; r < hi; ++r) {
                    const uint32_t kr = pkey[r];
                    less += kr < ki;
                    eq += kr == ki;
                }
            }
            if (eq == 1) {
                fin = lo + less;
            } else {
                const uint32_t di = m.id[i];
                for (int r = lo; r < hi; ++r) {
                    const uint32_t kr = pkey[r];
                    const int jj = m.ptmp[r];
                    const uint32_t dj = m.id[jj];
                    fin += (kr < ki) | ((kr == ki) & ((dj < di) | ((dj == di) & (jj < i))));
                }
            }
        }
        // the element goes straight to its sorted position: neighbouring
        // threads hold neighbouring buckets, so the writes stay close
        const int64_t go = o0 + fin;
        g.out_u[s][0][go] = m.us[0][i];
        g.out_u[s][1][go] = m.us[1][i];
        g.out_u[s][2][go] = m.us[2][i];
        g.out_id[s][go] = m.id[i];
        // the weight is not staged: read once more where the tile came from
        // (a sector this block has just read)
        if (g.out_w[s]) g.out_w[s][go] = t.rec ? rec_weight(t.rec + o0 + i) : t.w[t.input(o0 + i)];
    }
}

// A cell larger than the shared-memory capacity, ranked in global memory by
// the block: the cell's own part of the output arrays is the scratch, first
// for the keys and ids, then for the source position of every sorted place.
__device__ void sort_giant_cell(const SortGatherArgs& g, int s, const SortSrc& t, int64_t o, int64_t n, int32_t c)
{
    uint32_t* key = reinterpret_cast<uint32_t*>(g.out_u[s][0]) + o;
    uint32_t* id = g.out_id[s] + o;
    int32_t* src = g.out_cell[s] + o;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        if (t.rec) {
            key[i] = t.rec[o + i].key;
            id[i] = t.rec[o + i].id;
        } else {
            const uint32_t pid = t.id[t.input(o + i)];
            key[i] = g.draw.word0(s, pid);
            id[i] = pid;
        }
    }
    __syncthreads();
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) {
        const uint32_t ki = key[i], di = id[i];
        int64_t rank = 0;
        for (int64_t j = 0; j < n; ++j) {
            const uint32_t kj = key[j], dj = id[j];
            rank += (kj < ki) | ((kj == ki) & ((dj < di) | ((dj == di) & (j < i))));
        }
        src[rank] = (int32_t)i;
    }
    __syncthreads();
    for (int64_t p = threadIdx.x; p < n; p += blockDim.x) {
        const int64_t q = o + src[p];
        float x, y, z, wt = 0.0f;
        if (t.rec) {
            const SortRec r = t.rec[q];
            x = r.ux, y = r.uy, z = r.uz;
            id[p] = r.id;
            wt = rec_weight(&r);
        } else {
            const int64_t i = t.input(q);
            x = t.u[0][i], y = t.u[1][i], z = t.u[2][i];
            id[p] = t.id[i];
            if (g.out_w[s]) wt = t.w[i];
        }
        g.out_u[s][0][o + p] = x;
        g.out_u[s][1][o + p] = y;
        g.out_u[s][2][o + p] = z;
        if (g.out_w[s]) g.out_w[s][o + p] = wt;
        src[p] = c;
    }
    __syncthreads();
}

constexpr size_t kSortSmem = (size_t)kSortCap * (4 + 4 * kBucketsPerSlot + 4 + 12 + 2 + 2);
static_assert(kSortSmem <= 48 * 1024, "above what a launch may take without asking for it");

template <bool kChained>
__global__ void __launch_bounds__(kSortThreads, 10) k_sort_gather(const __grid_constant__ SortGatherArgs g)
{
    if (kChained) chain_start();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SortSmem m;
    m.id = reinterpret_cast<uint32_t*>(smem_raw);
    m.cnt = reinterpret_cast<int32_t*>(m.id + kSortCap);
    m.cmap = reinterpret_cast<uint32_t*>(m.cnt + kBucketsPerSlot * kSortCap);
    m.us[0] = reinterpret_cast<float*>(m.cmap + kSortCap);
    m.us[1] = m.us[0] + kSortCap;
    m.us[2] = m.us[1] + kSortCap;
    m.ptmp = reinterpret_cast<uint16_t*>(m.us[2] + kSortCap);
    m.pbk = m.ptmp + kSortCap;

    const int s = (int64_t)blockIdx.x < g.nb_e ? 0 : 1;
    const int64_t b = s == 0 ? blockIdx.x : blockIdx.x - g.nb_e;
    const int32_t* __restrict__ off = g.off[s];
    const int64_t c0 = g.stile[s][b];
    const int64_t c1 = g.stile[s][b + 1];
    if (c1 <= c0) return;
    const int64_t o0 = off[c0];
    const int64_t R = (int64_t)off[c1] - o0;
    if (R <= 0) return;

    SortSrc t;
    const SortSource source = sort_source(g.unsorted, s, g.n[s]);
    t.rec = source == kRecords ? g.rec[s] : nullptr;
    t.idx = source == kByIndex ? reinterpret_cast<const int32_t*>(g.rec[s]) : nullptr;
    t.id = g.in_id[s];
    for (int k = 0; k < 3; ++k) t.u[k] = g.in_u[s][k];
    t.w = g.in_w[s];

    if (R <= kSortCap) {
        sort_tile_block(g, s, t, m, c0, c1, o0, (int)R);
        return;
    }
    // A cell range larger than shared memory: runs of whole cells that fit
    // are sorted block-wide one after another; a cell above the capacity
    // alone is ranked in global memory.
    for (int64_t c = c0; c < c1;) {
        const int64_t o = off[c];
        if ((int64_t)off[c + 1] - o > kSortCap) {
            __syncthreads();
            sort_giant_cell(g, s, t, o, (int64_t)off[c + 1] - o, (int32_t)c);
            ++c;
            continue;
        }
        int64_t e = c + 1;
        while (e < c1 && (int64_t)off[e + 1] - o <= kSortCap) ++e;
        __syncthreads();
        sort_tile_block(g, s, t, m, c, e, o, (int)((int64_t)off[e] - o));
        c = e;
    }
}

// Tiles of the scan up to which k_scan_final adds up the tiles before its own
// (half a million cells; every block reads all the sums, 12 KB of them in the
// L2 there, and their number grows with the square).  301^2 cells, 89 tiles: the
// step 347 us with the block scan and launches one by one, 334 with the sums
// taken here and launches chained.
constexpr int64_t kOwnPrefixTiles = 512;

// CTAs per SM and species of the histogram (the launch's second
// grid dimension takes the two species), which runs in one wave of 1024-thread CTAs: 0.0394 ms on the 512^2 step against
// 0.0404 with four and 0.0435 with eight.
constexpr int kCountCtasPerSm = 2;

int grid_for(int64_t n, int threads, int max_blocks)
{
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (int)b;
}

}  // namespace

compton_status launch_bin_pairs(compton_ctx* ctx, const compton_species* e_in, const compton_species* g_in,
                                compton_species* e_out, compton_species* g_out, uint64_t step,
                                cudaStream_t stream)
{
    const int64_t C = ctx->cfg.n_cells;
    const int64_t ne = e_in->n, ng = g_in->n;
    const int64_t n_tiles = (C + kScanTile - 1) / kScanTile;
    const int64_t nmax = ne > ng ? ne : ng;
    const int64_t nb_e = (ne + kSortTile - 1) / kSortTile;
    const int64_t nb_g = (ng + kSortTile - 1) / kSortTile;
    // with per-particle weights a cell's density is its larger count; each
    // pair scales it by its own heavier weight
    const bool weighted = e_in->w_dev || g_in->w_dev;
    const compton_species* ins[2] = {e_in, g_in};
    compton_species* outs[2] = {e_out, g_out};
    ScanFinalArgs sf;
    sf.count_e = ctx->count[0];
    sf.count_g = ctx->count[1];
    sf.block_sums = ctx->block_sums;
    sf.n_tiles = n_tiles;
    sf.C = C;
    sf.n_e = ne;
    sf.n_g = ng;
    sf.off_e = ctx->off[0];
    sf.off_g = ctx->off[1];
    sf.cinfo = ctx->cinfo;
    sf.tile_cell = ctx->tile_cell;
    sf.stile_e = ctx->stile[0];
    sf.stile_g = ctx->stile[1];
    sf.nb_e = nb_e;
    sf.nb_g = nb_g;
    sf.n_pairs = ctx->n_pairs;
    sf.w_over_v = weighted ? 1.0 : ctx->cfg.w_over_v;
    const KeyDraw key_draw(ctx->cfg.seed, step, kStreamPairE, kStreamPairG);

    if (C <= kSmallCells && ne + ng <= kSmallParticles) {
        BinSmallArgs bs;
        for (int s = 0; s < 2; ++s) {
            bs.cell[s] = ins[s]->cell_dev;
            bs.idx[s] = reinterpret_cast<int32_t*>(ctx->rec[s]);
        }
        bs.scan = sf;
        bs.n_pairs = ctx->n_pairs;
        bs.unsorted = ctx->unsorted;
        bs.stats = ctx->stats;
        TimedScope ts_(ctx, COMPTON_K_COUNT, stream);
        launch_chained(k_bin_small, 1, kSmallThreads, 0, stream, bs);
        COMPTON_LAUNCH_CHECK(ctx, "k_bin_small");
    } else {
        // count[0], count[1] and unsorted lie in one block of the workspace
        COMPTON_CUDA_TRY(ctx, cudaMemsetAsync(ctx->count[0], 0,
                                              reinterpret_cast<char*>(ctx->unsorted + 4) -
                                                  reinterpret_cast<char*>(ctx->count[0]),
                                              stream));
        const dim3 cgrid(grid_for((nmax + 3) / 4, kCountThreads, ctx->n_sm * kCountCtasPerSm), 2);  // four per thread
        {
            TimedScope ts_(ctx, COMPTON_K_COUNT, stream);
            // a sixth of the positions begin a run, an eighth with the weight as one word more to gather
            const unsigned max_runs = weighted ? 16u : 24u;
            // 32-bit positions when the grid's last visited position fits
            const int64_t span = (nmax + 127) / 128 * 128 + (int64_t)cgrid.x * kCountThreads * 4;
            if (span < ((int64_t)1 << 31))
                launch_chained(k_count<int32_t>, cgrid, kCountThreads, 0, stream, e_in->cell_dev, ne, g_in->cell_dev,
                               ng, C, ctx->count[0], ctx->count[1], ctx->unsorted, max_runs, ctx->stats);
            else
                launch_chained(k_count<int64_t>, cgrid, kCountThreads, 0, stream, e_in->cell_dev, ne, g_in->cell_dev,
                               ng, C, ctx->count[0], ctx->count[1], ctx->unsorted, max_runs, ctx->stats);
        }
        COMPTON_LAUNCH_CHECK(ctx, "k_count");
        TimedScope scan_scope(ctx, COMPTON_K_SCAN, stream);
        launch_chained(k_scan_reduce, (unsigned)n_tiles, 256, 0, stream, ctx->count[0], ctx->count[1], C,
                       ctx->block_sums, n_tiles);
        COMPTON_LAUNCH_CHECK(ctx, "k_scan_reduce");
        if (n_tiles <= kOwnPrefixTiles) {
            launch_chained(k_scan_final<true>, (unsigned)n_tiles, 256, 0, stream, sf);
        } else {
            launch_chained(k_scan_blocks, 1, 1024, 0, stream, ctx->block_sums, n_tiles, ctx->n_pairs);
            COMPTON_LAUNCH_CHECK(ctx, "k_scan_blocks");
            launch_chained(k_scan_final<false>, (unsigned)n_tiles, 256, 0, stream, sf);
        }
        scan_scope.end();
        COMPTON_LAUNCH_CHECK(ctx, "k_scan_final");

        const dim3 pgrid(grid_for(nmax, kPlaceThreads, ctx->n_sm * kPlaceCtasPerSm), 2);
        PlaceArgs pa;
        for (int s = 0; s < 2; ++s) {
            pa.cell[s] = ins[s]->cell_dev;
            pa.id[s] = ins[s]->id_dev;
            pa.u[s][0] = ins[s]->ux_dev;
            pa.u[s][1] = ins[s]->uy_dev;
            pa.u[s][2] = ins[s]->uz_dev;
            pa.w[s] = ins[s]->w_dev;
            pa.n[s] = ins[s]->n;
            pa.off[s] = ctx->off[s];
            pa.cursor[s] = ctx->count[s];
            pa.rec[s] = ctx->rec[s];
        }
        pa.unsorted = ctx->unsorted;
        pa.C = C;
        pa.draw = key_draw;
        {
            TimedScope ts_(ctx, COMPTON_K_PLACE, stream);
            if ((int64_t)pgrid.x * pgrid.y <= chain_blocks(ctx))
                launch_chained(k_place<true>, pgrid, kPlaceThreads, 0, stream, pa);
            else
                k_place<false><<<pgrid, kPlaceThreads, 0, stream>>>(pa);
        }
        COMPTON_LAUNCH_CHECK(ctx, "k_place");
    }

    if (nb_e + nb_g > 0) {
        SortGatherArgs sg;
        for (int s = 0; s < 2; ++s) {
            sg.in_u[s][0] = ins[s]->ux_dev;
            sg.in_u[s][1] = ins[s]->uy_dev;
            sg.in_u[s][2] = ins[s]->uz_dev;
            sg.in_id[s] = ins[s]->id_dev;
            sg.in_w[s] = ins[s]->w_dev;
            sg.out_w[s] = ins[s]->w_dev ? outs[s]->w_dev : nullptr;
            sg.out_u[s][0] = outs[s]->ux_dev;
            sg.out_u[s][1] = outs[s]->uy_dev;
            sg.out_u[s][2] = outs[s]->uz_dev;
            sg.out_cell[s] = outs[s]->cell_dev;
            sg.out_id[s] = outs[s]->id_dev;
            sg.rec[s] = ctx->rec[s];
            sg.off[s] = ctx->off[s];
            sg.stile[s] = ctx->stile[s];
            sg.n[s] = ins[s]->n;
        }
        sg.draw = key_draw;
        sg.unsorted = ctx->unsorted;
        sg.nb_e = nb_e;
        const int smem = (int)kSortSmem;
        TimedScope ts_(ctx, COMPTON_K_SORT, stream);
        if (nb_e + nb_g <= chain_blocks(ctx))
            launch_chained(k_sort_gather<true>, (unsigned)(nb_e + nb_g), kSortThreads, smem, stream, sg);
        else
            k_sort_gather<false><<<(unsigned)(nb_e + nb_g), kSortThreads, smem, stream>>>(sg);
        COMPTON_LAUNCH_CHECK(ctx, "k_sort_gather");
    }
    return COMPTON_OK;
}

}  // namespace compton
