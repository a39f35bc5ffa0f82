// Streaming shuffle for populations of more than 16 models: the one-trip kernel's copies and block
// image (wash_shuffle_async.cuh), its serving arranged for permutations that fit no register.
//
// Shared memory (35 KB a block of 64 threads at N = 32 in fp32) leaves six blocks on an SM, so a block's
// life from its first copy to its last store decides the bandwidth, and registers are free.  What a
// selected coordinate costs is kept off that path: the warp lists its coordinates and draws the first
// 32 permutations while the copies are in flight, the Philox blocks dealt to all lanes
// (draw_permutations_by_warp); after the wait a lane per (coordinate, model) pair moves one value,
// which in [P][N] is one 128-byte store per coordinate.  Before, one lane drew a coordinate's eight blocks one
// after the other and moved its N values in a loop, all after the wait.  N = 32, fp32, 2^24 coordinates, [P][N],
// p = 0.01 / 0.03 / 0.1: 376 / 500 / 681 -> 334 / 373 / 482 us (reading and writing alone 331 / 338 / 361); [N][P] 415 / 599 / 753 ->
// 408 / 544 / 632 us; N = 20, bf16 + fp32, [P][N], p = 0.25: 1221 -> 678 us.
// [P][N] since then (move_quads, bulk copies), 2^23 coordinates: 169 / 191 / 233 -> 157 / 163 / 185 us.
#pragma once
#define WASH_SERVING_ONLY
#include "wash_shuffle_async.cuh"
#include "wash_bulk_copy.cuh"

namespace wash {

// [N][P]: up to this many coordinates of a round are moved by a lane per (coordinate, model) pair, more by a lane
// per coordinate: the models of a coordinate share a bank of the image.  N = 32, 2^24 coordinates: p = 0.01 (1.3
// coordinates a warp) 408 us by pairs, 422 by coordinates; p = 0.1 (12.8) 1155 / 627 us.
constexpr uint32_t kWidePairsMax = 6;

// What a (coordinate, model) pair's lane does: model n takes the value of model src.
template <class TA, class TB, int LAYOUT>
__device__ __forceinline__ void move_value(const ShuffleArgs &a, const unsigned char *image_a, const unsigned char *image_b, uint64_t g_block,
                                           uint32_t t_owner, uint32_t c, uint32_t n, uint32_t src)
{
    constexpr bool kHasB = TB::kCode != kDtypeNone;
    const int n_models = a.pop.N;
    const long long out = elem_index<LAYOUT>(a.pop, static_cast<int>(n), 4ll * static_cast<long long>(g_block + t_owner) + c);
    TA::store_elem(a.a, out, image_value<TA, LAYOUT>(image_a, n_models, a.pn_pad, t_owner, static_cast<int>(src), static_cast<int>(c)));
    if constexpr (kHasB) TB::store_elem(a.b, out, image_value<TB, LAYOUT>(image_b, n_models, a.pn_pad, t_owner, static_cast<int>(src), static_cast<int>(c)));
}

// Values of selected coordinates of a [P][N] image, four models to a thread (N a multiple of 4): model n of coordinate l takes the value of
// model byte n of perm + l * wide_pitch(N).  A word of the permutation, four values of the image and one store where a lane per (coordinate,
// model) pair read a byte, a value and stored 4 bytes; the issue slots of the moves, not the memory, were what kept the kernels from
// it.  Fixed points are stored, too (sectors are then written whole; alone that gave N = 32, p = 0.1 236 -> 226).  [P][N], pairs -> quads:
// shuffle_wide_kernel N = 20 fp32, 2^23 coordinates, p = 0.1 / 0.3 / 0.6 141 / 243 / 388 -> 127 / 201 / 297 us, N = 32 bf16 173 / 329 / 551 -> 151 / 256 /
// 405; shuffle_wide_pn_kernel N = 32 fp32 p = 0.01 / 0.1 / 0.6 170 / 234 / 693 -> 163 / 209 / 546, N = 64 346 / 544 / 1726 -> 334 / 491 / 1308.
template <class TA, class TB>
__device__ __forceinline__ uint32_t move_quads(const ShuffleArgs &a, const unsigned char *image_a, const unsigned char *image_b, uint64_t g_block,
                                               const uint32_t *s_perm, const uint8_t *s_entry, uint32_t count, uint32_t thread, uint32_t threads)
{
    constexpr bool kHasB = TB::kCode != kDtypeNone;
    const uint32_t n_models = static_cast<uint32_t>(a.pop.N), quads = n_models / 4u, group_elems = pn_group_elems(a.pop.N, a.pn_pad);
    uint32_t moved = 0;
    for (uint32_t i = thread; i < count * quads; i += threads) {
        const uint32_t l = (4u * i * a.pair_inverse) >> 20, q = i - l * quads;
        const uint32_t src = s_perm[l * wide_pitch(a.pop.N) + q], entry = s_entry[l], g = entry >> 2, c = entry & 3u;
        const uint32_t from = g * group_elems + c * n_models;
        const long long out = (4ll * static_cast<long long>(g_block + g) + c) * n_models + 4u * q;
        const uint32_t s0 = from + (src & 255u), s1 = from + ((src >> 8) & 255u), s2 = from + ((src >> 16) & 255u), s3 = from + (src >> 24);
        TA::store_group(static_cast<char *>(a.a) + out * TA::kBytes, TA::pack(TA::load_elem(image_a, s0), TA::load_elem(image_a, s1), TA::load_elem(image_a, s2), TA::load_elem(image_a, s3)));
        if constexpr (kHasB)
            TB::store_group(static_cast<char *>(a.b) + out * TB::kBytes, TB::pack(TB::load_elem(image_b, s0), TB::load_elem(image_b, s1), TB::load_elem(image_b, s2), TB::load_elem(image_b, s3)));
        moved += __popc(__vcmpne4(src, 0x03020100u + q * 0x04040404u)) >> 3;
    }
    return moved;
}

template <class TA, class TB, int LAYOUT, bool STAT>
__global__ void __launch_bounds__(64, 6) shuffle_wide_kernel(const __grid_constant__ ShuffleArgs a)
{
    await_previous();
    let_next_start();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr bool kHasB = TB::kCode != kDtypeNone;
    const int n_models = a.pop.N;
    const uint32_t T_ = blockDim.x, lane = threadIdx.x & 31u, warp_base = threadIdx.x & ~31u;
    // the images of the two stacks, the warps' lists, 32 permutations per warp
    const size_t group_elems = LAYOUT == kLayoutPN ? pn_group_elems(n_models, a.pn_pad) : 4u * static_cast<size_t>(n_models);
    unsigned char *image_a = smem_raw, *image_b = image_a + group_elems * T_ * TA::kBytes;
    uint8_t *list = image_b + (kHasB ? group_elems * T_ * TB::kBytes : 0) + 4 * warp_base;   // 128 bytes a warp: owner lane * 4 + coordinate slot
    uint32_t *s_perm = reinterpret_cast<uint32_t *>(image_b + (kHasB ? group_elems * T_ * TB::kBytes : 0) + 4 * T_) + warp_base * wide_pitch(n_models);

    const uint64_t g_block = a.group_lo + static_cast<uint64_t>(blockIdx.x) * T_;
    const uint32_t in_block = static_cast<uint32_t>(min(static_cast<uint64_t>(T_), a.group_hi - g_block));
    async_fetch<TA, LAYOUT>(smem_addr(image_a), a.a, a.pop, g_block, in_block, n_models, a.pn_pad);
    if constexpr (kHasB) async_fetch<TB, LAYOUT>(smem_addr(image_b), a.b, a.pop, g_block, in_block, n_models, a.pn_pad);

    uint32_t selected = 0, moved = 0, sel = 0;
    GroupInfo gi{0, 0, 0, 0, 0};
    if (threadIdx.x < in_block) {
        gi = find_group(a.pop, static_cast<uint32_t>(g_block + threadIdx.x), a.status);
        if (gi.thr != 0 && gi.valid != 0) {
            uint32_t m = 0xFu;   // a threshold of 2^32 selects whatever the word is
            if ((gi.thr >> 32) == 0) {
                const Philox4 w = philox4x32_10(gi.cgroup, gi.tensor_id, a.step_lo, a.step_hi8, a.keys);
                const uint32_t thr_lo = static_cast<uint32_t>(gi.thr);
                m = (w.x < thr_lo ? 1u : 0u) | (w.y < thr_lo ? 2u : 0u) | (w.z < thr_lo ? 4u : 0u) | (w.w < thr_lo ? 8u : 0u);
            }
            sel = m & ((1u << gi.valid) - 1u);   // coordinates beyond the tensor's end do not exist
        }
    }
    // the warp's selected coordinates, and the first 32 permutations, while the copies are in flight
    uint32_t total = 0;
    for (uint32_t left = sel, owners; (owners = __ballot_sync(0xFFFFFFFFu, left != 0)) != 0; left &= left - 1u) {
        if (left) list[total + __popc(owners & ((1u << lane) - 1u))] = static_cast<uint8_t>(lane * 4 + __ffs(left) - 1);
        total += __popc(owners);
    }
    __syncwarp();
    uint32_t entry = 0;
    auto draw = [&](uint32_t first, uint32_t count) {
        entry = lane < count ? list[first + lane] : 0u;
        const uint32_t owner = entry >> 2;
        const uint32_t cgroup = __shfl_sync(0xFFFFFFFFu, gi.cgroup, owner), tensor = __shfl_sync(0xFFFFFFFFu, gi.tensor_id, owner);
        draw_permutations_by_warp(s_perm, n_models, count, 4u * cgroup + (entry & 3u), tensor, a.step_lo, a.step_hi8, a.keys);
    };
    if (total) draw(0, min(32u, total));
    cp_async_wait_all();
    if (LAYOUT == kLayoutPN) __syncthreads();   // a group's bytes were copied by threads of other warps
    else __syncwarp();
    if constexpr (STAT) consensus_tile<TA, LAYOUT, 0>(a, image_a, gi, threadIdx.x < in_block);

    for (uint32_t first = 0; first < total; first += 32) {
        const uint32_t count = min(32u, total - first);
        if (first) draw(first, count);
        if (lane < count) ++selected;
        if (stored_together(LAYOUT, n_models) == 4) {
            const size_t skip = static_cast<size_t>(warp_base) * group_elems;
            moved += move_quads<TA, TB>(a, image_a + skip * TA::kBytes, image_b + skip * TB::kBytes, g_block + warp_base, s_perm, list + first, count, lane, 32u);
        } else if (LAYOUT == kLayoutPN || count <= kWidePairsMax) {
            // a lane per (coordinate, model) pair, the models of a coordinate side by side
            const uint32_t pairs = count * static_cast<uint32_t>(n_models);
            for (uint32_t base = 0; base < pairs; base += 32) {
                const uint32_t i = base + lane, l = min((i * a.pair_inverse) >> 20, count - 1u), n = i - l * static_cast<uint32_t>(n_models);
                const uint32_t its_entry = __shfl_sync(0xFFFFFFFFu, entry, l);
                if (i >= pairs) continue;
                const uint32_t src = reinterpret_cast<const uint8_t *>(s_perm + l * wide_pitch(n_models))[n];
                if (src == n) continue;
                move_value<TA, TB, LAYOUT>(a, image_a, image_b, g_block, warp_base + (its_entry >> 2), its_entry & 3u, n, src);
                ++moved;
            }
        } else if (lane < count) {
            // a lane per coordinate: the models of a coordinate lie a whole row apart here, and in one bank of the image
            const uint8_t *perm = reinterpret_cast<const uint8_t *>(s_perm + lane * wide_pitch(n_models));
#pragma unroll 4
            for (int n = 0; n < n_models; ++n) {
                const uint32_t src = perm[n];
                if (src == static_cast<uint32_t>(n)) continue;
                move_value<TA, TB, LAYOUT>(a, image_a, image_b, g_block, warp_base + (entry >> 2), entry & 3u, n, src);
                ++moved;
            }
        }
        __syncwarp();   // the permutations are overwritten by the next round
    }
    publish_block_stats(a.stats, a.stats_direct ? nullptr : a.stat_slots, selected, moved);
}

// [P][N] with a group of all models of kWideSplitBytes and more: two threads to a group, the block's selected
// coordinates in one list shared evenly by its warps.  Six blocks of 35 KB hold twice the warps that way,
// each with half the copies, draws and moves.  N = 32, fp32, 2^23 coordinates, p = 0.03 / 0.1 / 0.25: 197 / 246 / 410 us by the kernel
// above, 192 / 233 / 404 (both with a padded image at 0.25; without 357); N = 24, bf16 + fp32, p = 0.25 436 / 386; N = 64, fp32, p = 0.1 632 / 542.  Smaller groups (N = 20, fp32, p = 0.1
// 145 / 165 us) and [N][P] (N = 20 200 / 202, N = 17 bf16 103 / 162) lose more by the block's barriers;
// as they do with four models a thread (from 256 bytes on: N = 17 fp32, p = 0.1 121 / 134, N = 24 fp32 155 / 173, N = 32 bf16 151 / 171).
constexpr size_t kWideSplitBytes = 512;
// Coordinates whose permutations a warp of that kernel draws together.  The chain of swaps costs a warp the same for one coordinate and for
// 32, so few warps with many coordinates each take fewer instructions than an even share for all, and a longer way to the first
// move.  N = 32 fp32, 2^23, p = 0.1 / 0.3: an even share 226 / 407 us (by pairs), 16 209 / 349, 32 221 / 364.  The moves are dealt to all threads.
constexpr uint32_t kWideChunk = 16;

// BULK: the block's bytes come by one bulk copy a stack instead of 16 bytes a thread at a time, which are a sixth of the kernel's instructions
// (copies_in_bulk chooses).
template <class TA, class TB, bool BULK>
__global__ void __launch_bounds__(128, 6) shuffle_wide_pn_kernel(const __grid_constant__ ShuffleArgs a)
{
    await_previous();
    let_next_start();
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ uint32_t s_count, s_gave_up;
    __shared__ __align__(8) unsigned long long s_barrier;
    constexpr int LAYOUT = kLayoutPN;
    constexpr bool kHasB = TB::kCode != kDtypeNone;
    const int n_models = a.pop.N;
    const uint32_t groups = blockDim.x / 2u, lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
    // (pn_pad is 0 for these populations; left out of the kernel, the same one took 977 us for N = 32, 2^25 coordinates, p = 0.1, 963 with it)
    // the images of the two stacks, the block's list {coordinate within its tensor, tensor} and where it lies (group * 4 +
    // coordinate slot), as many permutations as the block has groups
    const uint32_t group_elems = pn_group_elems(n_models, a.pn_pad);
    unsigned char *image_a = smem_raw, *image_b = image_a + group_elems * groups * TA::kBytes;
    uint2 *s_key = reinterpret_cast<uint2 *>(image_b + (kHasB ? group_elems * groups * TB::kBytes : 0));
    uint32_t *s_perm = reinterpret_cast<uint32_t *>(s_key + 4 * groups);
    uint8_t *s_entry = reinterpret_cast<uint8_t *>(s_perm + groups * wide_pitch(n_models));

    const uint64_t g_block = a.group_lo + static_cast<uint64_t>(blockIdx.x) * groups;
    const uint32_t in_block = static_cast<uint32_t>(min(static_cast<uint64_t>(groups), a.group_hi - g_block));
    const uint32_t barrier = smem_addr(&s_barrier);
    if constexpr (BULK) {
        if (threadIdx.x == 0) {
            s_count = s_gave_up = 0;
            const uint32_t bytes_a = in_block * 4u * n_models * TA::kBytes, bytes_b = kHasB ? in_block * 4u * n_models * TB::kBytes : 0u;
            bulk_barrier_init(barrier);
            bulk_barrier_expect(barrier, bytes_a + bytes_b);
            bulk_copy(smem_addr(image_a), group_vec_ptr<TA, LAYOUT>(a.a, a.pop, g_block, 0), bytes_a, barrier);
            if constexpr (kHasB) bulk_copy(smem_addr(image_b), group_vec_ptr<TB, LAYOUT>(a.b, a.pop, g_block, 0), bytes_b, barrier);
        }
    } else {
        async_fetch<TA, LAYOUT>(smem_addr(image_a), a.a, a.pop, g_block, in_block, n_models, a.pn_pad);
        if constexpr (kHasB) async_fetch<TB, LAYOUT>(smem_addr(image_b), a.b, a.pop, g_block, in_block, n_models, a.pn_pad);
        if (threadIdx.x == 0) s_count = 0;
    }
    __syncthreads();

    uint32_t selected = 0, moved = 0;
    if (threadIdx.x < in_block) {
        const GroupInfo gi = find_group(a.pop, static_cast<uint32_t>(g_block + threadIdx.x), a.status);
        if (gi.thr != 0 && gi.valid != 0) {
            uint32_t m = 0xFu;   // a threshold of 2^32 selects whatever the word is
            if ((gi.thr >> 32) == 0) {
                const Philox4 w = philox4x32_10(gi.cgroup, gi.tensor_id, a.step_lo, a.step_hi8, a.keys);
                const uint32_t thr_lo = static_cast<uint32_t>(gi.thr);
                m = (w.x < thr_lo ? 1u : 0u) | (w.y < thr_lo ? 2u : 0u) | (w.z < thr_lo ? 4u : 0u) | (w.w < thr_lo ? 8u : 0u);
            }
            m &= (1u << gi.valid) - 1u;   // coordinates beyond the tensor's end do not exist
            if (m) {
                uint32_t pos = atomicAdd(&s_count, static_cast<uint32_t>(__popc(m)));
                for (; m; m &= m - 1u, ++pos) {
                    const uint32_t c = static_cast<uint32_t>(__ffs(m) - 1);
                    s_key[pos] = make_uint2(4u * gi.cgroup + c, gi.tensor_id);
                    s_entry[pos] = static_cast<uint8_t>(4u * threadIdx.x + c);
                }
            }
        }
    }
    __syncthreads();
    const uint32_t total = s_count;
    // a round: the permutations of up to `groups` coordinates, kWideChunk at a time by a warp
    auto draw = [&](uint32_t first) {
        const uint32_t in_round = min(groups, total - first);
        for (uint32_t at = ((warp + blockIdx.x) % warps) * kWideChunk; at < in_round; at += warps * kWideChunk) {
            const uint32_t count = min(kWideChunk, in_round - at);
            const uint2 key = s_key[first + at + min(lane, count - 1u)];
            draw_permutations_by_warp(s_perm + at * wide_pitch(n_models), n_models, count, key.x, key.y, a.step_lo, a.step_hi8, a.keys);
        }
        return in_round;
    };
    // the first round's permutations are drawn while the copies are in flight
    uint32_t in_round = draw(0);
    // (a group's bytes were copied, its permutations drawn by threads of other warps: both forms end with a barrier)
    if constexpr (BULK) {
        if (!block_copies_done(barrier, kBulkTries, &s_gave_up)) {   // (not seen) report and move nothing; the block stays for its copies once more as long
            if (threadIdx.x == 0) atomicOr(a.status, 8u);
            bulk_copies_done(barrier, kBulkTries);
            return;
        }
    } else {
        cp_async_wait_all();
        __syncthreads();
    }
    if (threadIdx.x == 0) selected = total;
    for (uint32_t first = 0; first < total;) {
        if (stored_together(LAYOUT, n_models) == 4) moved += move_quads<TA, TB>(a, image_a, image_b, g_block, s_perm, s_entry + first, in_round, threadIdx.x, blockDim.x);
        else {
            // a lane per (coordinate, model) pair, the models of a coordinate side by side
            for (uint32_t i = threadIdx.x; i < in_round * static_cast<uint32_t>(n_models); i += blockDim.x) {
                const uint32_t l = (i * a.pair_inverse) >> 20, n = i - l * static_cast<uint32_t>(n_models);
                const uint32_t src = reinterpret_cast<const uint8_t *>(s_perm + l * wide_pitch(n_models))[n];
                if (src == n) continue;
                const uint32_t entry = s_entry[first + l], g = entry >> 2, c = entry & 3u;
                const long long out = elem_index<LAYOUT>(a.pop, static_cast<int>(n), 4ll * static_cast<long long>(g_block + g) + c);
                const uint32_t from = g * group_elems + c * static_cast<uint32_t>(n_models) + src;
                TA::store_elem(a.a, out, TA::load_elem(image_a, from));
                if constexpr (kHasB) TB::store_elem(a.b, out, TB::load_elem(image_b, from));
                ++moved;
            }
        }
        first += in_round;
        if (first >= total) break;
        __syncthreads();   // the permutations are overwritten by the next round
        in_round = draw(first);
        __syncthreads();
    }
    publish_block_stats(a.stats, a.stats_direct ? nullptr : a.stat_slots, selected, moved);
}

template <class TA, class TB>
cudaError_t launch_shuffle_wide_typed(const ShuffleArgs &call, const LaunchShape &shape, cudaStream_t stream)
{
    constexpr bool kHasB = TB::kCode != kDtypeNone;
    ShuffleArgs args = call;
    args.pair_inverse = ((1u << 20) + static_cast<uint32_t>(args.pop.N) - 1u) / static_cast<uint32_t>(args.pop.N);
    const size_t group_elems = 4 * static_cast<size_t>(args.pop.N) + (args.pop.layout == kLayoutPN ? args.pn_pad : 0);
    const size_t per_thread = group_elems * (TA::kBytes + (kHasB ? TB::kBytes : 0)) + 4 + 4 * wide_pitch(args.pop.N);
    if (args.pop.layout == kLayoutPN && !args.sq.slots && 4 * static_cast<size_t>(args.pop.N) * (TA::kBytes + TB::kBytes) >= kWideSplitBytes) {
        // the images, the list (keys and places of every coordinate) and a permutation per group
        const size_t per_group = group_elems * (TA::kBytes + (kHasB ? TB::kBytes : 0)) + 4 * 8 + 4 + 4 * wide_pitch(args.pop.N);
        const uint32_t groups = per_group * 64 > 44 * 1024 ? 32 : 64;   // five blocks and more on an SM
        const size_t smem = (per_group * groups + 15) & ~static_cast<size_t>(15);
        auto kernel = copies_in_bulk(args, groups, TA::kBytes, TB::kBytes) ? shuffle_wide_pn_kernel<TA, TB, true> : shuffle_wide_pn_kernel<TA, TB, false>;
        KernelFit fit;
        cudaError_t err = kernel_fit(reinterpret_cast<const void *>(kernel), 2 * static_cast<int>(groups), smem, &fit);
        if (err != cudaSuccess) return err;
        if (fit.occupancy < 1) return cudaErrorLaunchOutOfResources;
        const uint64_t grid = (static_cast<uint64_t>(args.group_hi - args.group_lo) + groups - 1) / groups;
        if (grid == 0) return cudaSuccess;
        if (grid > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
        return launch_chained(kernel, static_cast<unsigned>(grid), 2 * groups, smem, stream, args);
    }
    int threads = shape.threads > 0 ? (shape.threads >= 64 ? 64 : 32) : 64;
    while (threads > 32 && per_thread * threads > 44 * 1024) threads >>= 1;   // five blocks and more on an SM
    const size_t smem = (per_thread * threads + 15) & ~static_cast<size_t>(15);
    const bool np = args.pop.layout == kLayoutNP;
    auto kernel = np ? shuffle_wide_kernel<TA, TB, kLayoutNP, false> : shuffle_wide_kernel<TA, TB, kLayoutPN, false>;
    if (args.sq.slots) kernel = np ? shuffle_wide_kernel<TA, TB, kLayoutNP, true> : shuffle_wide_kernel<TA, TB, kLayoutPN, true>;
    KernelFit fit;
    cudaError_t err = kernel_fit(reinterpret_cast<const void *>(kernel), threads, smem, &fit);
    if (err != cudaSuccess) return err;
    if (fit.occupancy < 1) return cudaErrorLaunchOutOfResources;
    const uint64_t grid = (static_cast<uint64_t>(args.group_hi - args.group_lo) + threads - 1) / threads;
    if (grid == 0) return cudaSuccess;
    if (grid > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    return launch_chained(kernel, static_cast<unsigned>(grid), threads, smem, stream, args);
}

inline cudaError_t launch_shuffle_wide(const ShuffleArgs &args, int a_dtype, int b_dtype, const LaunchShape &shape,
                                       cudaStream_t stream, bool *supported)
{
    *supported = true;
    if (a_dtype == kDtypeF32 && b_dtype == kDtypeNone) return launch_shuffle_wide_typed<F32, NoStack>(args, shape, stream);
    if (a_dtype == kDtypeBF16 && b_dtype == kDtypeNone) return launch_shuffle_wide_typed<BF16, NoStack>(args, shape, stream);
    if (a_dtype == kDtypeF32 && b_dtype == kDtypeF32) return launch_shuffle_wide_typed<F32, F32>(args, shape, stream);
    if (a_dtype == kDtypeBF16 && b_dtype == kDtypeF32) return launch_shuffle_wide_typed<BF16, F32>(args, shape, stream);
    if (a_dtype == kDtypeBF16 && b_dtype == kDtypeBF16) return launch_shuffle_wide_typed<BF16, BF16>(args, shape, stream);
    if (a_dtype == kDtypeF32 && b_dtype == kDtypeBF16) return launch_shuffle_wide_typed<F32, BF16>(args, shape, stream);
    *supported = false;
    return cudaSuccess;
}

}  // namespace wash
