// The shuffling step with one model per device: the worker form of Eq. 3.
//
// Every worker draws the same mask and the same permutations from the shared (seed, step),
// so only values cross the link.  Worker n owns a staging buffer; the selected coordinates
// with pi_i(n) != n take its slots in coordinate order and worker pi_i(n) stores its own
// value of the coordinate straight into the slot (a peer store when the buffer lives on
// another device).  After all workers have sent, each one copies its slots into its model.
//
// Work is cut into warp tiles of 128 groups (512 coordinates).  A block owns a contiguous range of warp
// tiles, the same one in all three kernels, so that "the slot of a coordinate" becomes the sum of
// the totals of the blocks before it plus a running count inside the block: no per-tile offsets are
// stored, only one total per block and column.
//   plan     draws the mask and, for selected coordinates, the permutation; writes a word per
//            four groups (low half: selected coordinates, high half: those whose new value comes
//            from another worker) and, per block, how many slots of every worker's buffer its
//            range takes (+ the selected count)
//   send     adds up the totals of the blocks before it (its first slots), then goes through its
//            range: lists the selected coordinates in order, a thread per coordinate redraws
//            the permutation, warp votes and the warps' counts number every
//            worker's slots, and this worker's value is stored where pi_i(n) is this worker
//   receive  the same replay for its own buffer only, from the high halves: no draw at all
// The plan reads no model data; send and receive touch only selected coordinates.
// All three kernels must be launched with the same grid (n_blocks).
//
// The plan is bound by the integer pipes (a Philox block per 4 coordinates), send and receive by the
// latency of a few dependent steps.  Five ResNet-50 models (25.6 M coordinates, 1.3e5 selected), parameters and
// momentum, launched back to back: plan 32 -> 21 us, a step 63.5 -> 45.1 us against a queue per warp, served 32 at a time, with
// mask words fetched one tile after the other and kernels that do not overlap; N = 32, 5.6e5 selected 205 -> 167 us.
#include "wash_device.cuh"
#include "wash_launch.cuh"
#include "wash_warp_tiles.cuh"
#include "wash_permutation.cuh"

namespace wash {

constexpr int kXThreads = 32 * kExchangeWarps;
static_assert(kExchangeTileGroups == kWarpTileGroups, "the exchange works on warp tiles");
constexpr uint32_t kNoDestination = 0xFFu;

// pi of coordinate `coord` of a tensor, as {need: bit n set iff pi(n) != n, dest: the n != self with
// pi(n) == self, if any}; nothing on inactive lanes.  Called by the whole warp, whose active lanes come
// first; s_perm: 32 * wide_pitch(N) words of the warp's own when N > 16.
__device__ __forceinline__ void routes_of(const ExchangeArgs &a, bool active, uint32_t coord, uint32_t tensor, uint32_t *s_perm,
                                          unsigned long long *need, uint32_t *dest)
{
    const int n_models = a.pop.N;
    unsigned long long nd = 0;
    uint32_t d = kNoDestination;
    if (n_models <= 16) {
        if (active) {
            uint64_t packed = draw_permutation_packed(n_models, coord, tensor, a.step_lo, a.step_hi8, a.keys);
            for (int n = 0; n < n_models; ++n, packed >>= 4) {
                const int src = static_cast<int>(static_cast<uint32_t>(packed) & 15u);
                if (src == n) continue;
                nd |= 1ull << n;
                if (src == a.self) d = static_cast<uint32_t>(n);
            }
        }
    } else {
        const uint32_t count = __popc(__ballot_sync(kFull, active));
        if (count) draw_permutations_by_warp(s_perm, n_models, count, coord, tensor, a.step_lo, a.step_hi8, a.keys);
        if (active) {
            const uint8_t *perm = reinterpret_cast<const uint8_t *>(s_perm + (threadIdx.x & 31u) * wide_pitch(n_models));
            for (int n = 0; n < n_models; ++n) {
                const int src = perm[n];
                if (src == n) continue;
                nd |= 1ull << n;
                if (src == a.self) d = static_cast<uint32_t>(n);
            }
        }
        __syncwarp();   // the permutations are overwritten by the next call
    }
    *need = nd;
    *dest = d;
}

// first and one-past-last warp tile of this block: the tiles are dealt out evenly, in order
__device__ __forceinline__ void block_range(const ExchangeArgs &a, uint32_t *t0, uint32_t *t1)
{
    *t0 = static_cast<uint32_t>(static_cast<uint64_t>(blockIdx.x) * a.n_wtiles / a.n_blocks);
    *t1 = static_cast<uint32_t>((static_cast<uint64_t>(blockIdx.x) + 1) * a.n_wtiles / a.n_blocks);
}

// A short row, a tile a warp: its three kernels leave room on the SMs and are bound by their starts, so each releases the next at
// once; on a long row waiting blocks are in the way of the running ones.  Plan, send and receive, all released at once / all after
// the wait / the plan alone at once: 2^17 coordinates, N = 20, p = 0.1 16.9 / 23.2 / 23.4 us; 2^20, N = 32, p = 0.1 39.2 / 40.5 / 58.5; 2^24,
// p = 0.01, N = 5 40.9 / 37.5, N = 64 166 / 134.
__device__ __forceinline__ bool short_row(const ExchangeArgs &a) { return a.n_wtiles <= a.n_blocks * static_cast<uint32_t>(kExchangeWarps); }

// The plan's block queue, as the sparse shuffle's: the coordinates its warps find, in any order (the
// counts do not depend on it), drawn a thread each when a piece of the range is done or the queue full.
constexpr uint32_t kPlanQueue = 1024;
// The mask words of up to so many warp tiles stay in shared memory until their selected coordinates are drawn: nothing is
// written before the first of these pieces is done, so the plan draws while the kernel before it (a step's receive, an
// optimizer) still runs, and the receive bits are set without a trip to the L2.  A step (plan, send, receive) against
// waiting first and writing word by word: ResNet-50 N = 5 47.0 -> 45.1 us (the plan alone 25.2 -> 21.0), N = 3 with 10^6
// coordinates 14.5 -> 9.4, 10^8 coordinates 220 -> 180.  Four blocks stay on an SM (28 KB a block, 45 at N = 64).
constexpr uint32_t kPlanHeldTiles = 128;

__global__ void __launch_bounds__(kXThreads, kExchangeBlocksPerSm) exchange_plan_kernel(const __grid_constant__ ExchangeArgs a)
{
    extern __shared__ uint32_t s_perm_all[];   // 32 * wide_pitch(N) words per warp when N > 16, else nothing
    __shared__ __align__(16) uint32_t s_words[32 * kPlanHeldTiles];
    __shared__ uint2 q_key[kPlanQueue];       // {coordinate within its tensor, tensor}
    __shared__ uint32_t q_elem[kPlanQueue];   // row element (rows are shorter than 2^32)
    __shared__ uint32_t s_total[kMaxN + 1], s_count;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const int n_models = a.pop.N, columns = n_models + 1;
    uint32_t *s_perm = s_perm_all + warp * 32u * wide_pitch(n_models);
    if (threadIdx.x < static_cast<uint32_t>(columns)) s_total[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_count = 0;
    uint32_t t_first, t_end;
    block_range(a, &t_first, &t_end);
    const bool release_early = short_row(a);
    if (release_early) let_next_start();
    const uint32_t pieces = (t_end - t_first + kPlanHeldTiles - 1u) / kPlanHeldTiles, per_piece = pieces ? (t_end - t_first + pieces - 1u) / pieces : 0u;
    LaneSegment ls;
    uint32_t p0 = t_first, p1;   // the piece's tiles
    do {
        p1 = min(p0 + per_piece, t_end);
        __syncthreads();
        uint32_t t = p0 + warp, sel = 0, sel_g0 = 0;   // sel: coordinates of the lane's last tile that are not queued yet; sel_g0: its first group there
        for (;;) {
            for (;;) {
                if (sel) {
                    uint32_t pos = atomicAdd(&s_count, static_cast<uint32_t>(__popc(sel)));
                    for (; sel && pos < kPlanQueue; sel &= sel - 1u, ++pos) {
                        const uint32_t bit = static_cast<uint32_t>(__ffs(sel) - 1), g = sel_g0 + (bit >> 2), c = bit & 3u;
                        if (g - ls.begin < ls.end - ls.begin) q_key[pos] = make_uint2(4u * (g + ls.cgroup_off) + c, ls.tensor);
                        else {
                            const GroupInfo gi = find_group(a.pop, g, a.status);
                            q_key[pos] = make_uint2(4u * gi.cgroup + c, gi.tensor_id);
                        }
                        q_elem[pos] = 4u * sel_g0 + bit;
                    }
                }
                if (sel || t >= p1) break;   // the queue is full, or the piece is done (lane by lane: nothing in this loop needs the warp together)
                sel_g0 = t * kExchangeTileGroups + 4u * lane;
                sel = lane_masks(a, sel_g0, a.pop.n_groups, ls);
                s_words[(t - p0) * 32u + lane] = sel;
                t += kExchangeWarps;
            }
            const bool again = __syncthreads_or(sel != 0 || t < p1);   // (orders the queue's entries and the mask words before the atomics below, too)
            const uint32_t count = min(s_count, kPlanQueue);
            for (uint32_t first = warp * 32u; first < count; first += kXThreads) {
                unsigned long long need;
                uint32_t dest;
                const bool active = first + lane < count;
                const uint2 key = active ? q_key[first + lane] : make_uint2(0, 0);
                routes_of(a, active, key.x, key.y, s_perm, &need, &dest);
                if ((need >> a.self) & 1ull) {
                    const uint32_t elem = q_elem[first + lane];
                    atomicOr(&s_words[(elem >> 4) - p0 * 32u], 0x10000u << (elem & 15u));
                }
                __syncwarp();
                uint32_t mine[2] = {0, 0};   // lane l counts workers l and l + 32
                for (int n = 0; n < n_models; ++n) {
                    const uint32_t votes = __popc(__ballot_sync(kFull, (need >> n) & 1ull));
                    if (lane == static_cast<uint32_t>(n & 31)) mine[n >> 5] = votes;
                }
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (mine[h]) atomicAdd(&s_total[lane + 32u * h], mine[h]);
                if (lane == 0) atomicAdd(&s_total[n_models], min(32u, count - first));
            }
            __syncthreads();   // the queue is free, the totals are complete
            if (threadIdx.x == 0) s_count = 0;
            if (!again) break;
            __syncthreads();
        }
        await_previous();
        if (!release_early) let_next_start();
        uint4 *out = reinterpret_cast<uint4 *>(a.mask + static_cast<size_t>(p0) * 32u);
        for (uint32_t i = threadIdx.x; i < (p1 - p0) * 8u; i += kXThreads) out[i] = reinterpret_cast<const uint4 *>(s_words)[i];
        p0 = p1;
    } while (p0 < t_end);
    if (threadIdx.x < static_cast<uint32_t>(columns)) a.block_total[static_cast<size_t>(blockIdx.x) * columns + threadIdx.x] = s_total[threadIdx.x];
}

__device__ __forceinline__ uint32_t load_element(const void *src, long long idx, int dtype)
{
    return dtype == kDtypeF32 ? F32::load_elem(src, idx) : BF16::load_elem(src, idx);
}
__device__ __forceinline__ void store_element(void *dst, long long idx, uint32_t bits, int dtype)
{
    if (dtype == kDtypeF32) F32::store_elem(dst, idx, bits);
    else BF16::store_elem(dst, idx, bits);
}

// Send and receive list the set bits of a block's mask words in order before they serve them, so that the
// few selected coordinates of many tiles share one round of a thread each.  Words lie in coordinate
// order and a thread takes two consecutive ones of a chunk of 16 warp tiles, so thread order is coordinate
// order.  Chunks are added until the list holds kListServe entries or the range ends.
constexpr uint32_t kChunkTiles = 2 * kExchangeWarps, kChunkCoords = kChunkTiles * 512;
constexpr uint32_t kListServe = 2048;

struct CoordList {
    uint32_t entry[kListServe + kChunkCoords];   // row elements (rows are shorter than 2^32)
    uint32_t warp_count[2][kExchangeWarps];
};

// this thread's words of the chunk that begins at tile t, nothing beyond tile t1
__device__ __forceinline__ uint2 chunk_words(const ExchangeArgs &a, uint32_t t, uint32_t t1)
{
    return t + threadIdx.x / 16u < t1 ? *reinterpret_cast<const uint2 *>(a.mask + static_cast<size_t>(t) * 32u + 2u * threadIdx.x) : make_uint2(0, 0);
}

// Lists bits of the mask words (kShift 0: selected, 16: received) from tile t on, at most up to tile t1, and moves t
// on; `words` are the next chunk's, fetched one chunk ahead.  Returns the length of the list.  Called by the
// whole block, which has left the previous list.
template <int kShift>
__device__ __forceinline__ uint32_t fill_list(const ExchangeArgs &a, CoordList &list, uint2 &words, uint32_t &t, uint32_t t1)
{
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t total = 0;
    for (uint32_t parity = 0; t < t1 && total < kListServe; t += kChunkTiles, parity ^= 1u) {
        uint32_t bits = ((words.x >> kShift) & 0xFFFFu) | ((words.y >> kShift) << 16);
        words = chunk_words(a, t + kChunkTiles, t1);
        uint32_t in_warp = 0;
        uint32_t pos = total + warp_exclusive_scan(__popc(bits), &in_warp);
        if (lane == 0) list.warp_count[parity][warp] = in_warp;
        __syncthreads();
#pragma unroll
        for (uint32_t w = 0; w < kExchangeWarps; ++w) {
            const uint32_t c = list.warp_count[parity][w];   // (rewritten two chunks, and a barrier, later)
            if (w < warp) pos += c;
            total += c;
        }
        const uint32_t elem = 4u * kExchangeTileGroups * t + 32u * threadIdx.x;
        for (; bits; bits &= bits - 1u, ++pos) list.entry[pos] = elem + static_cast<uint32_t>(__ffs(bits) - 1);
    }
    __syncthreads();
    return total;
}

__global__ void __launch_bounds__(kXThreads) exchange_send_kernel(const __grid_constant__ ExchangeArgs a)
{
    const bool release_early = short_row(a);
    if (release_early) let_next_start();
    await_previous();
    if (!release_early) let_next_start();
    extern __shared__ uint32_t s_perm_all[];
    __shared__ CoordList list;
    __shared__ uint32_t s_base[kMaxN], s_votes[kExchangeWarps][kMaxN];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const int n_models = a.pop.N, columns = n_models + 1;
    uint32_t *s_perm = s_perm_all + warp * 32u * wide_pitch(n_models);
    uint32_t t, t1;
    block_range(a, &t, &t1);
    uint2 words = chunk_words(a, t, t1);
    // slots of every worker's buffer taken before this block
    if (threadIdx.x < static_cast<uint32_t>(n_models)) s_base[threadIdx.x] = 0;
    __syncthreads();
    for (int col = 0; col < n_models; col += 8) {   // eight columns' loads in flight at a time
        uint32_t sum[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        for (uint32_t b = threadIdx.x; b < blockIdx.x; b += kXThreads) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (col + q < n_models) sum[q] += a.block_total[static_cast<size_t>(b) * columns + col + q];
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            sum[q] = __reduce_add_sync(kFull, sum[q]);
            if (lane == 0 && sum[q]) atomicAdd(&s_base[col + q], sum[q]);
        }
    }
    LaneSegment ls;
    while (t < t1) {
        const uint32_t total = fill_list<0>(a, list, words, t, t1);
        // rounds of a thread per coordinate: the warps vote worker by worker, the warps' counts turn
        // the votes into slots, then every thread with a destination copies its value
        for (uint32_t first = 0; first < total; first += kXThreads) {
            unsigned long long need;
            uint32_t dest, coord = 0, tensor = 0, value[2] = {0, 0};
            const bool active = first + threadIdx.x < total;
            if (active) {
                const uint32_t elem = list.entry[first + threadIdx.x], g = elem >> 2;
#pragma unroll
                for (int k = 0; k < 2; ++k)   // most values leave: fetched while the permutation is drawn
                    if (a.row[k]) value[k] = load_element(a.row[k], elem, a.dtype[k]);
                if (g - ls.begin >= ls.end - ls.begin) lane_segment_load(a, g, a.pop.n_groups, ls);
                coord = 4u * (g + ls.cgroup_off) + (elem & 3u);
                tensor = ls.tensor;
            }
            __syncwarp();
            routes_of(a, active, coord, tensor, s_perm, &need, &dest);
            uint32_t before = 0;   // slots of worker `dest` taken by the lanes before this one
            for (int n = 0; n < n_models; ++n) {
                const uint32_t votes = __ballot_sync(kFull, (need >> n) & 1ull);
                if (dest == static_cast<uint32_t>(n)) before = __popc(votes & ((1u << lane) - 1u));
                if (lane == static_cast<uint32_t>(n & 31)) s_votes[warp][n] = __popc(votes);
            }
            __syncthreads();
            if (dest != kNoDestination) {
                uint32_t slot = s_base[dest] + before;
                for (uint32_t w = 0; w < warp; ++w) slot += s_votes[w][dest];
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if (!a.row[k]) continue;
                    if (static_cast<long long>(slot) < a.capacity[k]) store_element(a.staging[k][dest], slot, value[k], a.dtype[k]);
                    else atomicOr(a.status, 4u);   // staging buffer too small: nothing is written beyond it
                }
            }
            __syncthreads();
            if (threadIdx.x < static_cast<uint32_t>(n_models)) {
                uint32_t sum = 0;
#pragma unroll
                for (uint32_t w = 0; w < kExchangeWarps; ++w) sum += s_votes[w][threadIdx.x];
                s_base[threadIdx.x] += sum;
            }
            __syncthreads();
        }
    }
}

__global__ void __launch_bounds__(kXThreads) exchange_receive_kernel(const __grid_constant__ ExchangeArgs a)
{
    const bool release_early = short_row(a);
    if (release_early) let_next_start();
    await_previous();
    if (!release_early) let_next_start();
    __shared__ CoordList list;
    __shared__ uint32_t s_part[kExchangeWarps];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const int columns = a.pop.N + 1;
    uint32_t t, t1;
    block_range(a, &t, &t1);
    uint2 words = chunk_words(a, t, t1);
    if (a.stats && blockIdx.x == 0 && warp < 2) {   // the step's totals: selected coordinates, values this worker receives
        const int col = warp == 0 ? a.pop.N : a.self;
        uint32_t sum = 0;
        for (uint32_t b = lane; b < a.n_blocks; b += 32) sum += a.block_total[static_cast<size_t>(b) * columns + col];
        sum = __reduce_add_sync(kFull, sum);
        if (lane == 0) atomicAdd(a.stats + warp, static_cast<unsigned long long>(sum));
    }
    // slots of this worker's buffer taken before this block
    {
        uint32_t sum = 0;
#pragma unroll 4
        for (uint32_t b = threadIdx.x; b < blockIdx.x; b += kXThreads) sum += a.block_total[static_cast<size_t>(b) * columns + a.self];
        sum = __reduce_add_sync(kFull, sum);
        if (lane == 0) s_part[warp] = sum;
    }
    __syncthreads();
    uint32_t base = 0;
#pragma unroll
    for (int w = 0; w < kExchangeWarps; ++w) base += s_part[w];
    const void *src[2] = {a.row[0] ? a.staging[0][a.self] : nullptr, a.row[1] ? a.staging[1][a.self] : nullptr};
    while (t < t1) {
        const uint32_t total = fill_list<16>(a, list, words, t, t1);
        for (uint32_t i = threadIdx.x; i < total; i += kXThreads) {
            const uint32_t slot = base + i, elem = list.entry[i];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                if (!a.row[k]) continue;
                if (static_cast<long long>(slot) < a.capacity[k]) store_element(a.row[k], elem, load_element(src[k], slot, a.dtype[k]), a.dtype[k]);
                else atomicOr(a.status, 4u);
            }
        }
        base += total;
        __syncthreads();   // the list is rewritten
    }
}

// Populations above 16 models keep their permutations in shared memory: with the kernels' static
// shared memory that is more than the default 48 KiB per block, so the kernel's limit is raised first.
static cudaError_t perm_smem(const ExchangeArgs &args, const void *kernel, size_t *bytes)
{
    *bytes = args.pop.N > 16 ? 4u * kXThreads * wide_pitch(args.pop.N) : 0;
    if (*bytes == 0) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(4u * kXThreads * wide_pitch(kMaxN)));
}

cudaError_t launch_exchange_plan(const ExchangeArgs &args, cudaStream_t stream)
{
    if (args.n_blocks == 0) return cudaSuccess;
    size_t smem = 0;
    cudaError_t err = perm_smem(args, reinterpret_cast<const void *>(exchange_plan_kernel), &smem);
    if (err != cudaSuccess) return err;
    return launch_chained(exchange_plan_kernel, args.n_blocks, kXThreads, smem, stream, args);
}

cudaError_t launch_exchange_send(const ExchangeArgs &args, cudaStream_t stream)
{
    if (args.n_blocks == 0) return cudaSuccess;
    size_t smem = 0;
    cudaError_t err = perm_smem(args, reinterpret_cast<const void *>(exchange_send_kernel), &smem);
    if (err != cudaSuccess) return err;
    return launch_chained(exchange_send_kernel, args.n_blocks, kXThreads, smem, stream, args);
}

cudaError_t launch_exchange_receive(const ExchangeArgs &args, cudaStream_t stream)
{
    if (args.n_blocks == 0) return cudaSuccess;
    return launch_chained(exchange_receive_kernel, args.n_blocks, kXThreads, 0, stream, args);
}

}  // namespace wash
