// Sparse shuffle (WASH_MODE_SPARSE): the mask is drawn first, without touching the stacks, and
// only the selected coordinates are loaded, permuted and stored -- the paper's point that a
// step moves p d values, not d, carried onto one GPU.
//
// A block walks a contiguous range of warp tiles (wash_warp_tiles.cuh), its warps taking turns.
// The selected coordinates of all its warps go to one queue in shared memory; when the range is
// done (or the queue full) the block serves the queue: a thread per coordinate draws the
// permutation, then a thread per (coordinate, model) pair moves one value, so that neither step
// runs on a few lanes of every warp and all the loads of a set are in flight at once.
//
// The exchange is in place: a warp loads all values of its set of coordinates before it stores
// the first of them.
//
// Two costs.  The mask: one Philox block per 4 coordinates on the integer pipes (2^27 coordinates:
// 80 us for the blocks alone, 86 us with the compares, this kernel 92 us at N = 2, p = 1e-4).  The
// values: DRAM serves about 45e9 isolated 4-byte loads a second, 22e9 stores and 20e9 pairs
// of both (measured, one access per 800 bytes), 1 us per 20 000 moved values and stack.  That is the rate of isolated accesses
// and no bound for denser ones, which share DRAM pages and sectors: ResNet-50 N = 8, bf16 + fp32, p = 5e-3 (1.8e6 values in
// both stacks) would take 90 us by it and takes 70.  With a queue per warp, served at the end of the warp's
// range by a lane per coordinate, and launches that do not overlap, the same took (before -> now): that one 89.1 -> 77.1,
// ResNet-18 N = 5 with momentum, p = 1e-3 21.0 -> 10.5, ResNet-50 N = 10 with momentum, p = 0.01 -> 0 70.8 -> 56.1, 2^27 coordinates N = 2
// at p = 1e-3 119 -> 97.5 us.
#pragma once
#include <cmath>
#include "wash_device.cuh"
#include "wash_launch.cuh"
#include "wash_warp_tiles.cuh"
#include "wash_permutation.cuh"

namespace wash {

constexpr int kSparseWarps = 4;
constexpr int kSparseThreads = 32 * kSparseWarps;
constexpr int kSparsePairs = 4;      // (coordinate, model) pairs a lane has in flight
// Shares of the coordinates from which [N][P] is served a lane per coordinate (serve_row): pairs take 128 / N neighbouring
// coordinates of a model side by side, half a sector at N = 32, a lane per coordinate 32, but all N values one
// after the other.  fp32, pairs / rows: N = 8, 2^25, 10 % 331 / 323, 30 % 483 / 411 us; N = 16, 2^24, 10 % 375 / 390, 30 % 518 / 407; N = 20 30 %
// 710 / 686; N = 24, 2^23, 2 % 146 / 177, 5 % 266 / 277; N = 28 2 % 173 / 216, 10 % 421 / 389; N = 32, 2^24, 1 % 266 / 265, 10 % 1417 / 901, all
// 5830 / 1927; N = 5 30 % 338 / 421.
constexpr float kRowsShare = 0.25f, kRowsShareLarge = 0.06f;   // 8 to 23 models, 24 and more
// Selected values per coordinate (of all models and stacks) up to which the next kernel may start at once: while masks
// are most of the time, the next launch of this kernel draws its own beside this one's last; where values are, its waiting blocks
// are in the way.  Back to back, released early / after the wait: N = 2, 2^23 coordinates, p = 1e-3 (0.002) 7.4 / 9.1 us, ResNet-18 N = 5 with
// momentum (0.01) 10.5 / 12.7, N = 5, 2^23, p = 0.01 (0.05) 10.2 / 12.4, ResNet-50 N = 5, p = 0.05 -> 0 (0.12) 42.7 / 45.6; N = 20, 2^20, p = 0.01 (0.2)
// 9.2 / 7.2, N = 32, 2^20, p = 0.01 (0.32) 23.5 / 16.6, N = 5, 2^20, p = 0.1 (0.5) 8.7 / 6.0.
constexpr double kReleaseShare = 0.15;
constexpr double kSparsePerBlock = 16.0;   // selected coordinates a block expects, at least

// entries of the queue: a permutation of up to 16 models stays in its entry (8 bytes), a larger one
// takes wide_pitch(N) words beside it.  Half as many from 29 models on: eight blocks would leave the L1 28 KB and the sectors that
// neighbouring coordinates share would not stay (6.3e6 coordinates, 1 %: N = 28 85 us, 29 113, 33 with 256 entries 97).
__host__ __device__ constexpr uint32_t sparse_queue_capacity(int n_models) { return n_models <= 28 ? 512u : 256u; }

// A scattered value of a stack.  HALF_LINE: the L2 is asked to fetch 64 bytes around it instead of the 128 it fetches otherwise
// (it does not go below 64).  Where accesses are dense enough for the bytes to count, and not the memory's pages alone, that
// is a third of the loads' time: 2^21 loads of 4 bytes, one in 800 / 200 / 80 bytes 45 / 40 / 28 us, with 64 bytes 41 / 26 / 22.
template <class T, bool HALF_LINE>
__device__ __forceinline__ uint32_t load_scattered(const void *stack, long long idx)
{
    if constexpr (!HALF_LINE) return T::load_elem(stack, idx);
    const void *p = static_cast<const char *>(stack) + idx * T::kBytes;
    uint32_t v;
    if constexpr (T::kBytes == 4) asm volatile("ld.global.L2::64B.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    else {
        uint16_t h;
        asm volatile("ld.global.L2::64B.u16 %0, [%1];" : "=h"(h) : "l"(p) : "memory");
        v = h;
    }
    return v;
}

// list of a warp of the form for dense selections: a tile's 512 coordinates and what the tile before left
constexpr uint32_t kWarpList = 512 + 32;

struct SparseArgs {
    ShuffleArgs s;
    uint32_t n_wtiles;      // warp tiles in [group_lo, group_hi)
    uint32_t per_block, extra;   // tiles of a block: per_block, one more in the first `extra` blocks
    bool release_early;     // the next kernel may start with this one's masks
    uint32_t in_set;        // coordinates whose N values a warp moves at a time: 32 * kSparsePairs / N
    uint32_t column_offset; // ROWS: where the lanes' columns lie in shared memory
    uint32_t inverse;       // 2^16 / d, rounded up, for the division of a pair's number (below 128) by in_set ([N][P]) or N ([P][N])
};

// One stack's values of a lane's coordinate: all loaded into the lane's column of shared memory, then stored.
template <class T, int LAYOUT, bool HALF_LINE, class PERM>
__device__ __forceinline__ void serve_row(const PopView &pop, void *stack, uint32_t *column, long long elem, const PERM &source_of)
{
    const int n_models = pop.N;
#pragma unroll 8
    for (int n = 0; n < n_models; ++n) column[n * kSparseThreads] = load_scattered<T, HALF_LINE>(stack, elem_index<LAYOUT>(pop, n, elem));
#pragma unroll 4
    for (int n = 0; n < n_models; ++n) {
        const uint32_t src = source_of(n);
        if (src != static_cast<uint32_t>(n)) T::store_elem(stack, elem_index<LAYOUT>(pop, n, elem), column[src * kSparseThreads]);
    }
}

// MIRROR: the moved values go to a second copy of the stacks as well (wash_step_host: the caller's buffers).
// ROWS: a lane per coordinate loads all its values before it stores them (serve_row), instead of a lane per (coordinate,
// model) pair.
template <class TA, class TB, int LAYOUT, bool MIRROR, bool ROWS, bool HALF_LINE>
__global__ void __launch_bounds__(kSparseThreads, 32 / kSparseWarps) shuffle_sparse_kernel(const __grid_constant__ SparseArgs p)
{
    if (p.release_early) let_next_start();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint32_t s_count;
    constexpr bool kHasB = TB::kCode != kDtypeNone;
    const ShuffleArgs &a = p.s;
    const int n_models = a.pop.N;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t capacity = sparse_queue_capacity(n_models);
    // [entry: {coordinate within its tensor, tensor}, then the packed permutation][entry: row element,
    // counted from the first element of the block's range][N > 16: byte n of entry e's permutation at word e * wide_pitch(N)]
    uint2 *q_key = reinterpret_cast<uint2 *>(smem_raw);
    uint32_t *q_elem = reinterpret_cast<uint32_t *>(q_key + capacity);
    uint32_t *q_wide = q_elem + capacity;
    if (threadIdx.x == 0) s_count = 0;

    const uint32_t t_first = blockIdx.x * p.per_block + min(blockIdx.x, p.extra);
    const uint32_t t_end = t_first + p.per_block + (blockIdx.x < p.extra ? 1u : 0u);
    const uint32_t block_group = a.group_lo + t_first * kWarpTileGroups;
    const long long block_elem = 4ll * static_cast<long long>(block_group);

    __syncthreads();

    uint32_t selected = 0, moved = 0;
    LaneSegment ls;
    uint32_t t = t_first + warp, sel = 0, sel_g0 = 0;   // sel: coordinates of the lane's last tile that are not queued yet; sel_g0: its first group there
    for (;;) {
        for (;;) {
            if (sel) {
                uint32_t pos = atomicAdd(&s_count, static_cast<uint32_t>(__popc(sel)));
                for (; sel && pos < capacity; sel &= sel - 1u, ++pos) {
                    const uint32_t bit = static_cast<uint32_t>(__ffs(sel) - 1), g = sel_g0 + (bit >> 2), c = bit & 3u;
                    if (g - ls.begin < ls.end - ls.begin) q_key[pos] = make_uint2(4u * (g + ls.cgroup_off) + c, ls.tensor);
                    else {
                        const GroupInfo gi = find_group(a.pop, g, a.status);
                        q_key[pos] = make_uint2(4u * gi.cgroup + c, gi.tensor_id);
                    }
                    q_elem[pos] = 4u * (sel_g0 - block_group) + bit;
                }
            }
            if (sel || t >= t_end) break;   // the queue is full, or the range is done (lane by lane: nothing in this loop needs the warp together)
            sel_g0 = a.group_lo + t * kWarpTileGroups + 4u * lane;
            sel = lane_masks(a, sel_g0, a.group_hi, ls);
            t += kSparseWarps;
        }
        const bool again = __syncthreads_or(sel != 0 || t < t_end);   // (orders the queue's entries, too)
        const uint32_t count = min(s_count, capacity);
        await_previous();   // the masks read nothing but the tables; the stacks come now
        if (!p.release_early) let_next_start();
        if (n_models <= 16) {
            for (uint32_t e = threadIdx.x; e < count; e += kSparseThreads) {
                const uint2 key = q_key[e];
                const uint64_t packed = draw_permutation_packed(n_models, key.x, key.y, a.step_lo, a.step_hi8, a.keys);
                q_key[e] = make_uint2(static_cast<uint32_t>(packed), static_cast<uint32_t>(packed >> 32));
                ++selected;
            }
        } else {
            for (uint32_t first = warp * 32u; first < count; first += kSparseThreads) {
                const uint32_t in_round = min(32u, count - first);
                const uint2 key = q_key[first + min(lane, in_round - 1u)];
                draw_permutations_by_warp(q_wide + first * wide_pitch(n_models), n_models, in_round, key.x, key.y, a.step_lo, a.step_hi8, a.keys);
                if (lane < in_round) ++selected;
            }
        }
        __syncthreads();
        if constexpr (ROWS) {
            uint32_t *column = reinterpret_cast<uint32_t *>(smem_raw + p.column_offset) + threadIdx.x;
            for (uint32_t e = threadIdx.x; e < count; e += kSparseThreads) {
                const long long elem = block_elem + q_elem[e];
                const uint2 packed = q_key[e];
                const uint8_t *wide = reinterpret_cast<const uint8_t *>(q_wide + e * wide_pitch(n_models));
                const auto source_of = [&](int n) -> uint32_t { return n_models <= 16 ? ((n < 8 ? packed.x : packed.y) >> (4 * (n & 7))) & 15u : wide[n]; };
                serve_row<TA, LAYOUT, HALF_LINE>(a.pop, a.a, column, elem, source_of);
                if constexpr (kHasB) serve_row<TB, LAYOUT, HALF_LINE>(a.pop, a.b, column, elem, source_of);
                for (int n = 0; n < n_models; ++n) moved += source_of(n) != static_cast<uint32_t>(n) ? 1u : 0u;
            }
        } else {
            // the lane's pairs of a set: [N][P] takes neighbouring coordinates of one model side by side,
            // [P][N] the models of one coordinate
            uint32_t pair_entry[kSparsePairs], pair_model[kSparsePairs];
#pragma unroll
            for (int k = 0; k < kSparsePairs; ++k) {
                const uint32_t i = lane + 32u * k, outer = (i * p.inverse) >> 16;
                const uint32_t inner = i - outer * (LAYOUT == kLayoutNP ? p.in_set : static_cast<uint32_t>(n_models));
                pair_entry[k] = LAYOUT == kLayoutNP ? inner : outer;
                pair_model[k] = LAYOUT == kLayoutNP ? outer : inner;
                if (pair_model[k] >= static_cast<uint32_t>(n_models) || pair_entry[k] >= p.in_set) pair_entry[k] = 0xFFFFu;   // no pair
            }
            for (uint32_t first = warp * p.in_set; first < count; first += kSparseWarps * p.in_set) {
                const uint32_t left = count - first;
                uint32_t va[kSparsePairs], vb[kSparsePairs];
                long long out[kSparsePairs];
#pragma unroll
                for (int k = 0; k < kSparsePairs; ++k) {
                    out[k] = -1;
                    if (pair_entry[k] < left) {
                        const uint32_t e = first + pair_entry[k], n = pair_model[k];
                        uint32_t src;
                        if (n_models <= 16) {
                            const uint2 packed = q_key[e];
                            src = ((n < 8 ? packed.x : packed.y) >> (4u * (n & 7u))) & 15u;
                        } else src = reinterpret_cast<const uint8_t *>(q_wide + e * wide_pitch(n_models))[n];
                        if (src != n) {
                            const long long elem = block_elem + q_elem[e];
                            const long long in = elem_index<LAYOUT>(a.pop, static_cast<int>(src), elem);
                            out[k] = elem_index<LAYOUT>(a.pop, static_cast<int>(n), elem);
                            va[k] = load_scattered<TA, HALF_LINE>(a.a, in);
                            if constexpr (kHasB) vb[k] = load_scattered<TB, HALF_LINE>(a.b, in);
                        }
                    }
                }
                __syncwarp();   // every value of the set is loaded before the first is overwritten
#pragma unroll
                for (int k = 0; k < kSparsePairs; ++k) {
                    if (out[k] < 0) continue;
                    TA::store_elem(a.a, out[k], va[k]);
                    if constexpr (kHasB) TB::store_elem(a.b, out[k], vb[k]);
                    if constexpr (MIRROR) {
                        TA::store_elem(a.mirror_a, out[k], va[k]);
                        if constexpr (kHasB) TB::store_elem(a.mirror_b, out[k], vb[k]);
                    }
                    ++moved;
                }
            }
        }
        if (!again) break;
        __syncthreads();   // the queue is free
        if (threadIdx.x == 0) s_count = 0;
        __syncthreads();
    }
    publish_block_stats(a.stats, a.stats_direct ? nullptr : a.stat_slots, selected, moved);
}

// Where much is selected: a warp by itself, without the block's barriers.  It lists a tile's selected coordinates in order behind
// the few left over from the tile before and serves them 32 at a time, a lane per coordinate (serve_row), so that
// one warp's mask, another's loads and a third one's stores run beside each other all the time.
template <class TA, class TB, int LAYOUT, bool HALF_LINE>
__global__ void __launch_bounds__(kSparseThreads, 32 / kSparseWarps) shuffle_sparse_warps_kernel(const __grid_constant__ SparseArgs p)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr bool kHasB = TB::kCode != kDtypeNone;
    const ShuffleArgs &a = p.s;
    const int n_models = a.pop.N;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    // [a list per warp: row elements, counted from the first of the warp's range][a column of N words per thread][N > 16: 32 permutations per warp]
    uint32_t *list = reinterpret_cast<uint32_t *>(smem_raw) + warp * kWarpList;
    uint32_t *columns = reinterpret_cast<uint32_t *>(smem_raw) + kSparseWarps * kWarpList;
    uint32_t *column = columns + threadIdx.x, *s_perm = columns + n_models * kSparseThreads + warp * 32u * wide_pitch(n_models);

    const uint64_t range = blockIdx.x * kSparseWarps + warp, ranges = static_cast<uint64_t>(gridDim.x) * kSparseWarps;
    const uint32_t t_first = static_cast<uint32_t>(range * p.n_wtiles / ranges), t_end = static_cast<uint32_t>((range + 1) * p.n_wtiles / ranges);
    const uint32_t first_group = a.group_lo + t_first * kWarpTileGroups;
    uint32_t selected = 0, moved = 0, length = 0;
    LaneSegment ls, served;
    bool waited = false;
    for (uint32_t t = t_first; t < t_end; ++t) {
        const uint32_t g0 = a.group_lo + t * kWarpTileGroups + 4u * lane;
        uint32_t sel = lane_masks(a, g0, a.group_hi, ls), in_tile = 0;
        uint32_t pos = length + warp_exclusive_scan(__popc(sel), &in_tile);
        for (; sel; sel &= sel - 1u, ++pos) list[pos] = 4u * (g0 - first_group) + static_cast<uint32_t>(__ffs(sel) - 1);
        length += in_tile;
        __syncwarp();
        if (length < 32u && t + 1 < t_end) continue;
        if (!waited) {   // the masks read nothing but the tables; the stacks come now
            await_previous();
            let_next_start();
            waited = true;
        }
        uint32_t done = 0;
        while (length - done >= 32u || (t + 1 == t_end && done < length)) {
            const uint32_t count = min(32u, length - done);
            const bool active = lane < count;
            const long long elem = 4ll * first_group + list[done + min(lane, count - 1u)];
            const uint32_t g = static_cast<uint32_t>(elem >> 2);
            if (g - served.begin >= served.end - served.begin) lane_segment_load(a, g, a.group_hi, served);
            const uint32_t coord = 4u * (g + served.cgroup_off) + static_cast<uint32_t>(elem & 3);
            __syncwarp();
            uint64_t packed = 0;
            if (n_models > 16) draw_permutations_by_warp(s_perm, n_models, count, coord, served.tensor, a.step_lo, a.step_hi8, a.keys);
            else if (active) packed = draw_permutation_packed(n_models, coord, served.tensor, a.step_lo, a.step_hi8, a.keys);
            if (active) {
                const uint8_t *wide = reinterpret_cast<const uint8_t *>(s_perm + lane * wide_pitch(n_models));
                const auto source_of = [&](int n) -> uint32_t { return n_models <= 16 ? static_cast<uint32_t>(packed >> (4 * n)) & 15u : wide[n]; };
                serve_row<TA, LAYOUT, HALF_LINE>(a.pop, a.a, column, elem, source_of);
                if constexpr (kHasB) serve_row<TB, LAYOUT, HALF_LINE>(a.pop, a.b, column, elem, source_of);
                for (int n = 0; n < n_models; ++n) moved += source_of(n) != static_cast<uint32_t>(n) ? 1u : 0u;
                ++selected;
            }
            __syncwarp();
            done += count;
        }
        const uint32_t rest = length - done;   // fewer than 32: to the front of the list
        const uint32_t keep = lane < rest ? list[done + lane] : 0u;
        __syncwarp();
        if (lane < rest) list[lane] = keep;
        length = rest;
        __syncwarp();
    }
    if (!waited) {   // a block's end without the wait would let later kernels pass the one before this
        await_previous();
        let_next_start();
    }
    publish_block_stats(a.stats, a.stats_direct ? nullptr : a.stat_slots, selected, moved);
}

// Which selections shuffle_sparse_warps_kernel serves.  Time by pairs (by rows of the block's queue: r) / by warps:
//   [P][N], one stack: a lane takes a coordinate's N neighbouring values itself, so where most of them move the queue's
//     reading per pair is what it saves.  2^24 coordinates, fp32: N = 3 20 % 77 / 86, 30 % 110 / 105, all 258 / 228; 4 15 % 78 / 75, 2^27 10 %
//     450 / 430; 5 20 % 106 / 120, 30 % 147 / 145, 50 % 210 / 187; 8 20 % 138 / 133, all 511 / 368; 10 30 % 251 / 231; 12 30 % 283 / 293,
//     50 % 422 / 393; 14 (2^23) 50 % 254 / 288, all 440 / 388; 16 all 954 / 1197.  N = 2 2^24 10 % 44 / 43, 20 % 59 / 64, 30 % 90 / 83,
//     2^27 8 % 272 / 256, 10 % 343 / 289, 20 % 470 / 440.
//     bf16: N = 2 10 % 43 / 40, 3 15 % 56 / 57, 5 20 % 93 / 98, 30 % 136 / 118, 8 30 % 184 / 203, 50 % 281 / 223, 10 50 % 358 / 361, all 646 / 449.
//     Two stacks by pairs throughout (N = 7 all 281 / 294, N = 5 407 / 403).
//   [N][P]: from 18 models on in between, where pairs fill a fraction of a sector and rows wait for the block; with the shared
//     memory held to kWarpsCarveout so that the L1 keeps the sectors that neighbouring coordinates share (N = 20, 15 %, 2^23 333 us without, 280
//     with; 32 509 / 407; a larger L1 yet loses resident warps, 270 and 435).  N = 18 6 % 192 / 197, 15 % 244 / 235, 30 % r 308 / 281;
//     20 15 % 280 / 280, 30 % r 346 / 284, 50 % r 390 / 368; 24 6 % 295 / 260, 15 % r 363 / 301, 50 % r 454 / 448; 32 6 % r 402 / 348,
//     30 % r 557 / 489, 50 % r 627 / 673; 48 6 % r 582 / 534, 15 % r 763 / 692, 30 % r 817 / 934; 64 15 % r 1019 / 958, 30 % r 1109 / 1410;
//     bf16 + fp32 20 15 % 599 / 450, 24 30 % r 638 / 540.
constexpr int kWarpsCarveout = 132 * 100 / 228;   // per cent of the largest shared memory
inline bool sparse_by_warps(const ShuffleArgs &args, bool bf16, bool two_stacks)
{
    const int N = args.pop.N;
    const float share = args.expected_share;
    if (args.pop.layout == kLayoutNP) return N >= 18 && share >= (N < 40 ? 0.05f : 0.025f) && share < (N < 40 ? 0.4f : 0.12f);
    if (two_stacks) return false;
    if (bf16) return N <= 12 && share >= (N <= 3 ? 0.1f : N <= 6 ? 0.25f : N <= 9 ? 0.4f : 0.7f);
    if (N == 2 && args.pop.n_groups >= 1u << 24) return share >= 0.08f;
    if (N == 4 || N == 8) return share >= 0.15f;   // a coordinate's values are whole 16-byte pieces
    return N <= 15 && share >= (N <= 3 ? 0.25f : N <= 10 ? 0.3f : N <= 12 ? 0.4f : 0.7f);
}

template <class TA, class TB>
cudaError_t launch_shuffle_sparse_typed(const ShuffleArgs &args, const LaunchShape &shape, cudaStream_t stream)
{
    if (args.group_hi <= args.group_lo) return cudaSuccess;
    SparseArgs p;
    p.s = args;
    const bool by_warp = sparse_by_warps(args, TA::kBytes == 2, TB::kCode != kDtypeNone);
    const bool half = fetch_half_lines(args, by_warp, TA::kBytes, TB::kBytes);
    p.n_wtiles = (args.group_hi - args.group_lo + kWarpTileGroups - 1) / kWarpTileGroups;
    size_t smem = sparse_queue_capacity(args.pop.N) * (12 + (args.pop.N > 16 ? 4 * static_cast<size_t>(wide_pitch(args.pop.N)) : 0));
    const bool np = args.pop.layout == kLayoutNP;
    auto kernel = np ? shuffle_sparse_kernel<TA, TB, kLayoutNP, false, false, false> : shuffle_sparse_kernel<TA, TB, kLayoutPN, false, false, false>;
    if (half) kernel = np ? shuffle_sparse_kernel<TA, TB, kLayoutNP, false, false, true> : shuffle_sparse_kernel<TA, TB, kLayoutPN, false, false, true>;
    if (args.mirror_a) kernel = np ? shuffle_sparse_kernel<TA, TB, kLayoutNP, true, false, false> : shuffle_sparse_kernel<TA, TB, kLayoutPN, true, false, false>;
    else if (np && args.expected_share >= (args.pop.N >= 24 ? kRowsShareLarge : args.pop.N >= 8 ? kRowsShare : 2.f)) {
        kernel = half ? shuffle_sparse_kernel<TA, TB, kLayoutNP, false, true, true> : shuffle_sparse_kernel<TA, TB, kLayoutNP, false, true, false>;
        p.column_offset = static_cast<uint32_t>(smem);
        smem += 4 * static_cast<size_t>(args.pop.N) * kSparseThreads;
    }
    if (!args.mirror_a && by_warp) {
        auto by_warps = np ? shuffle_sparse_warps_kernel<TA, TB, kLayoutNP, false> : shuffle_sparse_warps_kernel<TA, TB, kLayoutPN, false>;
        if (half && np) by_warps = shuffle_sparse_warps_kernel<TA, TB, kLayoutNP, true>;
        smem = 4 * kSparseWarps * static_cast<size_t>(kWarpList) + 4 * static_cast<size_t>(args.pop.N) * kSparseThreads +
               (args.pop.N > 16 ? 4 * static_cast<size_t>(wide_pitch(args.pop.N)) * kSparseThreads : 0);
        KernelFit fit;
        cudaError_t err = kernel_fit(reinterpret_cast<const void *>(by_warps), kSparseThreads, smem, &fit);
        if (err == cudaSuccess && np) err = cudaFuncSetAttribute(reinterpret_cast<const void *>(by_warps), cudaFuncAttributePreferredSharedMemoryCarveout, kWarpsCarveout);
        if (err != cudaSuccess) return err;
        if (fit.occupancy < 1) return cudaErrorLaunchOutOfResources;
        // four waves, as far as a warp keeps two tiles: ranges that select unequally even out
        const uint32_t wave = static_cast<uint32_t>(shape.sm_count > 0 ? shape.sm_count : 148) * static_cast<uint32_t>(fit.occupancy);
        uint32_t grid = p.n_wtiles / (2 * kSparseWarps);
        if (grid > 4 * wave) grid = 4 * wave;
        if (grid < wave) grid = wave;
        const uint32_t want = (p.n_wtiles + kSparseWarps - 1) / kSparseWarps;
        if (grid > want) grid = want;
        return launch_chained(by_warps, grid, kSparseThreads, smem, stream, p);
    }
    KernelFit fit;
    cudaError_t err = kernel_fit(reinterpret_cast<const void *>(kernel), kSparseThreads, smem, &fit);
    if (err != cudaSuccess) return err;
    if (fit.occupancy < 1) return cudaErrorLaunchOutOfResources;
    const uint32_t resident = static_cast<uint32_t>(shape.sm_count > 0 ? shape.sm_count : 148) * static_cast<uint32_t>(fit.occupancy);
    // Grid.  A block costs its start, its barriers and its end (about 1.5 us of a resident slot), so it takes as many tiles
    // as it can; what ends that is the serving: several waves let one block's (memory-bound) serving overlap the
    // next one's (multiply-bound) mask.  So: whole waves, as many as keep a block's expected selection at what [N][P]
    // serves in 400 scattered values (300 in two stacks or more than 8 models), [P][N] in 300 coordinates, but not
    // below kSparsePerBlock coordinates and 2 ([P][N] 3) tiles a warp.  Measured (blocks of 2 or 3 tiles a warp throughout ->
    // this rule): N = 2, 2^27 coordinates, p = 3e-3 / 0.01 / 0.03 134 / 162 / 198 -> 106 / 124 / 183 us, 2^25, p = 0.01 41.2 -> 31.9; N = 3,
    // 2.5e7, p = 3e-3 26.8 -> 20.9; ResNet-50 N = 5, p = 0.05 -> 0 44.9 -> 42.7; [P][N] N = 8, 2^25, p = 0.01 43.3 -> 36.7, N = 16, p = 3e-3
    // 39.9 -> 31.7.  A larger load loses where values are many (400 instead of 300 for ResNet-50 N = 8 bf16 + fp32, p = 5e-3: 79.4
    // against 77.1, N = 20, p = 2e-3 51.6 against 50.3), a broken wave where waves are few ([P][N] N = 8, 2^25: 1.4 waves
    // 41.9, two 38.8).  Half a wave where that serves everything and the next kernel is released at once (half_wave_serves).
    const bool one_stack = TB::kCode == kDtypeNone;
    const double expected = static_cast<double>(args.expected_share) * 4.0 * static_cast<double>(args.group_hi - args.group_lo);
    double by_tiles = static_cast<double>(p.n_wtiles) / (kSparseWarps * (np ? 2 : 3));
    // (one tile a warp where the queue would overflow: [P][N] N = 5, 2^25, p = 0.15 183 -> 172 us, [N][P] p = 0.1 194 -> 184)
    if (expected > by_tiles * (np ? 0.75 : 1.0) * sparse_queue_capacity(args.pop.N)) by_tiles = static_cast<double>(p.n_wtiles) / kSparseWarps;
    const double load = np ? (one_stack && args.pop.N <= 8 ? 400.0 : 300.0) / args.pop.N : 300.0;   // coordinates of a block, one stack
    p.release_early = static_cast<double>(args.expected_share) * args.pop.N * (one_stack ? 1 : 2) <= kReleaseShare;
    const double by_load = expected * (one_stack ? 1.0 : 2.0) / load;
    uint32_t grid = static_cast<uint32_t>(fmin(fmin(expected / kSparsePerBlock, by_tiles), resident * ceil(by_load / resident)));
    if (grid < resident) grid = p.release_early && half_wave_serves(args.pop.layout, args.pop.N, one_stack ? 1 : 2, expected, by_load, resident, p.n_wtiles) ? resident / 2 : resident;
    const uint32_t want = (p.n_wtiles + kSparseWarps - 1) / kSparseWarps;
    if (grid > want) grid = want;
    p.per_block = p.n_wtiles / grid;
    p.extra = p.n_wtiles % grid;
    p.in_set = 32u * kSparsePairs / static_cast<uint32_t>(args.pop.N);
    const uint32_t divisor = args.pop.layout == kLayoutNP ? p.in_set : static_cast<uint32_t>(args.pop.N);
    p.inverse = (65536u + divisor - 1u) / divisor;
    return launch_chained(kernel, grid, kSparseThreads, smem, stream, p);
}

inline cudaError_t launch_shuffle_sparse_tiles(const ShuffleArgs &args, int a_dtype, int b_dtype, const LaunchShape &shape,
                                               cudaStream_t stream, bool *supported)
{
    *supported = true;
    if (a_dtype == kDtypeF32 && b_dtype == kDtypeNone) return launch_shuffle_sparse_typed<F32, NoStack>(args, shape, stream);
    if (a_dtype == kDtypeBF16 && b_dtype == kDtypeNone) return launch_shuffle_sparse_typed<BF16, NoStack>(args, shape, stream);
    if (a_dtype == kDtypeF32 && b_dtype == kDtypeF32) return launch_shuffle_sparse_typed<F32, F32>(args, shape, stream);
    if (a_dtype == kDtypeBF16 && b_dtype == kDtypeF32) return launch_shuffle_sparse_typed<BF16, F32>(args, shape, stream);
    if (a_dtype == kDtypeBF16 && b_dtype == kDtypeBF16) return launch_shuffle_sparse_typed<BF16, BF16>(args, shape, stream);
    if (a_dtype == kDtypeF32 && b_dtype == kDtypeBF16) return launch_shuffle_sparse_typed<F32, BF16>(args, shape, stream);
    *supported = false;
    return cudaSuccess;
}

}  // namespace wash
