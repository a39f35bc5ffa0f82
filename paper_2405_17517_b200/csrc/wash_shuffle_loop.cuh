// Streaming shuffle for populations whose group of all models is small (N * 16 bytes in fp32):
// a resident grid of one-warp blocks, each walking tiles of 32 * G groups with two shared-memory
// stages.
//
// With one group per thread and one trip per thread (wash_shuffle_async.cuh) a thread spends a
// few hundred instructions around its single group -- block start, table lookup, the copies'
// addresses, the statistics' block reduction -- which is nothing beside 320 bytes of a ten-model
// group but fills the issue slots at 40 % of the memory bandwidth when the group has 32 bytes.
// Here a warp stays: the copies of its next tile are started, the mask of the current tile is
// drawn while they travel, the current tile (whose copies were started one trip earlier) is
// served, and the table entry, the counters and the launch constants live in registers across
// trips.  Tiles are dealt round-robin over the blocks, so the blocks resident at one moment read
// neighbouring addresses.
//
// Serving costs a hundred issue slots and more on a mostly idle warp however few coordinates it
// serves (a permutation is a Philox block and a chain of swaps), so it is done once a tile for the
// G groups of every lane together: the tile's selected coordinates are listed and dealt to the
// lanes 32 at a time.  Bound: HBM up to p = 1e-3, issue slots above it.  N = 2, fp32, 2^27 coordinates
// (before: two groups per lane, served one after the other, and a flush kernel for the counters):
// p = 1e-2 390 -> 245 us, 1e-3 206 -> 203; 2^25 coordinates: p = 0.1 134 -> 95, 0.02 125 -> 71; one model
// step of N = 3, 2^20 coordinates 12.3 -> 8.3.
//
// As issue slots bound it, the tile kernel is also compiled for each population of 2 to 5 models, whose copies,
// swap chains and row addresses then need no loop control or multiplications (run-time N -> compiled in: N = 2,
// 2^27 coordinates p = 1e-2 236 -> 216 us, 1e-3 205 -> 195; 2^25 coordinates: N = 2 [P][N] p = 0.1 94.0 -> 81.0, N = 3
// p = 1e-2 85.4 -> 82.4 (bf16 78.6 -> 70.4), N = 4 bf16 88.9 -> 79.9, N = 5 144.7 -> 137.9; N = 3, 2^20 7.49 -> 7.07).
// Larger populations move more bytes for the same control.  The narrow form (two groups a lane) likewise: 2^27 coordinates,
// p = 1e-4, N = 2 174 -> 170, bf16 205 -> 169, N = 3 257 -> 248, bf16 223 -> 198; N = 5 bf16, 2^24, 34.9 -> 32.7.
//
// An image of a stage is the one-trip kernel's block image with T = 32 (the block is one warp,
// so every helper of that kernel -- copies, serving, padding rule -- is used as it is).
#pragma once
#define WASH_SERVING_ONLY
#include "wash_shuffle_async.cuh"

namespace wash {

__device__ __forceinline__ void cp_async_commit()
{
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int K>
__device__ __forceinline__ void cp_async_wait_all_but_latest()   // all groups of copies but the K latest
{
    asm volatile("cp.async.wait_group %0;" ::"n"(K) : "memory");
}

// The table entry of the lane's previous group; a group of the same segment needs no lookup.
struct SegCache {
    uint32_t begin, end;   // groups [begin, end) of the row
    uint32_t tensor_id, cgroup_begin, numel, seg;
    uint32_t thr_lo;       // the threshold's low word
    uint32_t thr_hi;       // 1: the threshold is 2^32 (every coordinate selected)
    uint32_t plain;        // groups of the segment that hold four coordinates, 0 unless 0 < threshold < 2^32
};

__device__ __forceinline__ GroupInfo find_group_cached(const PopView &pop, SegCache &sc, uint32_t g, uint32_t *status)
{
    if (g - sc.begin >= sc.end - sc.begin) {
        uint32_t s = __ldg(pop.tile_first + (g >> kTileShift));
        const uint32_t last = static_cast<uint32_t>(pop.n_seg) - 1u;
        while (s < last && g >= __ldg(&pop.seg[s].group_end)) ++s;
        const uint4 lo = __ldg(reinterpret_cast<const uint4 *>(pop.seg + s));
        const uint4 hi = __ldg(reinterpret_cast<const uint4 *>(pop.seg + s) + 1);
        if (g < lo.x || g >= lo.y) {   // table inconsistent with the row: report, touch nothing
            if (status) atomicOr(status, 1u);
            return GroupInfo{0, 0, 0, 0, s};
        }
        const bool drawn = hi.w == 0 && hi.z != 0;   // 0 < threshold < 2^32: the mask words decide
        sc = SegCache{lo.x, lo.y, lo.z, lo.w, hi.x, s, hi.z, hi.w, drawn ? min(hi.x >> 2, lo.y - lo.x) : 0u};
    }
    const uint32_t local = g - sc.begin;
    GroupInfo gi;
    gi.seg = sc.seg;
    gi.tensor_id = sc.tensor_id;
    gi.cgroup = sc.cgroup_begin + local;
    gi.thr = static_cast<uint64_t>(sc.thr_lo) | (static_cast<uint64_t>(sc.thr_hi) << 32);
    // coordinates of the tensor from this group on; the segment may end in a group of padding only
    const long long left = static_cast<long long>(sc.numel) - 4ll * local;
    gi.valid = left >= 4 ? 4 : (left > 0 ? static_cast<int>(left) : 0);
    return gi;
}

// Starts the copies of the full tile of 32 * G groups that begins at group g_first into a stage.
// fp32 only: [N][P]: lane l copies the vector of every model for its G groups; [P][N] without
// padding: the tile's bytes are contiguous and are copied as they lie, 512 bytes per warp and copy.
template <int LAYOUT, int G>
__device__ __forceinline__ void fetch_full_tile_f32(uint32_t image, uint32_t image_stride, const void *base, const PopView &pop,
                                                    uint32_t g_first, int n_models)
{
    const uint32_t lane = threadIdx.x;
    if (LAYOUT == kLayoutNP) {
        const size_t row_bytes = static_cast<size_t>(pop.padded_P) * 4;
        const char *src0 = static_cast<const char *>(base) + (static_cast<size_t>(g_first) + lane) * 16;
        uint32_t dst0 = image + lane * 16;
#pragma unroll
        for (int i = 0; i < G; ++i, src0 += 512, dst0 += image_stride) {
            const char *src = src0;
            uint32_t dst = dst0;
            for (int j = 0; j < n_models; ++j, src += row_bytes, dst += 512) cp_async<16>(dst, src);
        }
    } else {
        const char *src = static_cast<const char *>(base) + (static_cast<size_t>(g_first) * n_models + lane) * 16;
        uint32_t dst0 = image + lane * 16;
#pragma unroll
        for (int i = 0; i < G; ++i, dst0 += image_stride) {
            uint32_t dst = dst0;
            for (int j = 0; j < n_models; ++j, src += 512, dst += 512) cp_async<16>(dst, src);
        }
    }
}

// The tile's selected coordinates, listed as owner lane * 4G + bit, where bit 4 i + c stands for
// coordinate c of the lane's group of image i.  `sel` has at most 4G bits.  Returns their number.
template <int G>
__device__ __forceinline__ uint32_t list_selected(uint16_t *list, uint32_t sel)
{
    const uint32_t lane = threadIdx.x;
    uint32_t total = 0;
    for (uint32_t owners = __ballot_sync(0xFFFFFFFFu, sel != 0); owners; owners = __ballot_sync(0xFFFFFFFFu, sel != 0)) {
        if (sel) list[total + __popc(owners & ((1u << lane) - 1u))] = static_cast<uint16_t>(lane * (4 * G) + __ffs(sel) - 1);
        sel &= sel - 1u;
        total += __popc(owners);
    }
    __syncwarp();
    return total;
}

// kN: the population size where it is compiled in (the helpers read it from the arguments: the assumption reaches
// them), 0 = run-time N.
template <class TA, class TB, int LAYOUT, int G, int kN, int FORM>
__global__ void __launch_bounds__(32, G == 2 ? 32 : 28) shuffle_loop_kernel(const __grid_constant__ ShuffleArgs a)
{
    if constexpr (kN != 0) __builtin_assume(a.pop.N == kN);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr bool kHasB = TB::kCode != kDtypeNone;
    constexpr uint32_t T_ = 32;   // the launch has one warp per block
    const int n_models = kN ? kN : a.pop.N;
    const uint32_t lane = threadIdx.x;
    const size_t group_elems = LAYOUT == kLayoutPN ? pn_group_elems(n_models, a.pn_pad) : 4u * static_cast<size_t>(n_models);
    const uint32_t a_bytes = static_cast<uint32_t>(group_elems * T_ * TA::kBytes);
    const uint32_t b_bytes = kHasB ? static_cast<uint32_t>(group_elems * T_ * TB::kBytes) : 0u;
    const uint32_t stage_bytes = G * (a_bytes + b_bytes);
    uint16_t *s_list = reinterpret_cast<uint16_t *>(smem_raw + 2 * stage_bytes);   // the tile's selected coordinates

    // group indices fit 32 bits (the table holds them so); a tile index therefore too
    const uint32_t n_tiles = static_cast<uint32_t>((a.group_hi - a.group_lo + T_ * G - 1) / (T_ * G));
    const uint32_t full_tiles = static_cast<uint32_t>((a.group_hi - a.group_lo) / (T_ * G));   // the tiles before the ragged one
    const uint32_t group_lo = static_cast<uint32_t>(a.group_lo);
    const uint32_t image0 = smem_addr(smem_raw);
    // starts the copies of a tile into a stage (nothing beyond the last tile) and closes their group
    auto fetch = [&](uint32_t tile, uint32_t stage) {
        const uint32_t g_first = group_lo + tile * (T_ * G);
        constexpr bool kFastA = TA::kBytes == 4, kFastB = !kHasB || TB::kBytes == 4;
        const bool linear = LAYOUT == kLayoutNP || a.pn_pad == 0;
        if (tile < full_tiles && linear && (kFastA || kFastB)) {
            const uint32_t image_a = image0 + stage * stage_bytes;
            if constexpr (kFastA) fetch_full_tile_f32<LAYOUT, G>(image_a, a_bytes + b_bytes, a.a, a.pop, g_first, n_models);
            if constexpr (kHasB && TB::kBytes == 4) fetch_full_tile_f32<LAYOUT, G>(image_a + a_bytes, a_bytes + b_bytes, a.b, a.pop, g_first, n_models);
        }
        if (tile < n_tiles && !(tile < full_tiles && linear && kFastA && kFastB)) {
#pragma unroll 1
            for (int i = 0; i < G; ++i) {
                const uint64_t g_block = static_cast<uint64_t>(g_first) + static_cast<uint64_t>(i) * T_;
                if (g_block >= a.group_hi) break;
                const uint32_t in_tile = static_cast<uint32_t>(min(static_cast<uint64_t>(T_), a.group_hi - g_block));
                const uint32_t image_a = image0 + stage * stage_bytes + i * (a_bytes + b_bytes);
                if (!(tile < full_tiles && linear && kFastA)) async_fetch<TA, LAYOUT>(image_a, a.a, a.pop, g_block, in_tile, n_models, a.pn_pad);
                if constexpr (kHasB)
                    if (!(tile < full_tiles && linear && TB::kBytes == 4)) async_fetch<TB, LAYOUT>(image_a + a_bytes, a.b, a.pop, g_block, in_tile, n_models, a.pn_pad);
            }
        }
        cp_async_commit();
    };

    uint32_t selected = 0, moved = 0, stage = 0;
    SegCache sc{0, 0, 0, 0, 0, 0, 0, 0, 0};
    uint32_t tile = blockIdx.x;
    // A launch of one tile a warp draws its masks, which need nothing but the tables, before it waits for the kernel before it.
    // (With several tiles the copies of the first come first: they hide the masks.)  With the counters' single report
    // (publish_warp_stats), call after call, p = 0.01: N = 3, 2^20 coordinates 7.1 -> 4.3 us, 2^17 5.6 -> 4.1; N = 2, 2^20 8.0 -> 4.2; several tiles a
    // warp, by the report alone: N = 2, 2^22 12.5 -> 10.9, N = 5, 2^21 11.0 -> 9.4.  Of these the early masks are the part that takes a kernel of this library
    // before it.  Neither / the report alone / both, call after call | behind an elementwise kernel of another library on other data | on the stacks
    // (the device's time, the host ahead): N = 3, 2^20 7.2 5.5 3.7 | 7.6 6.1 6.0 | 6.2 4.1 4.1;  2^17 5.7 4.0 2.8 | 5.1 4.1 4.1 | 4.1 3.1 3.7;  N = 2, 2^20 8.0 6.4 4.1 | 6.2 4.2 4.2 |
    // 6.2 5.3 4.6.
    const bool one_trip = n_tiles <= gridDim.x;
    if (!one_trip) {
        await_previous();
        let_next_start();
        fetch(tile, 0);
    }
    for (; tile < n_tiles; tile += gridDim.x, stage ^= 1u) {
        const uint32_t next = tile + gridDim.x;
        if (!one_trip) fetch(next >= tile ? next : n_tiles, stage ^ 1u);   // beyond the last tile (also when the index wraps) a fetch copies nothing
        const uint32_t g_first = group_lo + tile * (T_ * G);
        uint32_t sel = 0;   // bit 4 i + c: coordinate c of group g_first + 32 i + lane
        // the usual tile: full, every lane's G groups whole and in the segment of its previous
        // group, thresholds that the mask words decide -- then nothing is looked up or predicated
        const uint32_t local = g_first + lane - sc.begin;
        if (tile < full_tiles && __all_sync(0xFFFFFFFFu, local < sc.plain && local + (G - 1) * T_ < sc.plain)) {
            uint32_t w[4 * G];
#pragma unroll
            for (int i = 0; i < G; ++i) {
                const Philox4 block = philox4x32_10(sc.cgroup_begin + local + i * T_, sc.tensor_id, a.step_lo, a.step_hi8, a.keys);
                w[4 * i] = block.x;
                w[4 * i + 1] = block.y;
                w[4 * i + 2] = block.z;
                w[4 * i + 3] = block.w;
            }
            sel = pack_below(w, sc.thr_lo);
        } else {
#pragma unroll 1
            for (int i = 0; i < G; ++i) {
                const uint64_t g = static_cast<uint64_t>(g_first) + static_cast<uint64_t>(i) * T_ + lane;
                if (g >= a.group_hi) break;
                const GroupInfo gi = find_group_cached(a.pop, sc, static_cast<uint32_t>(g), a.status);
                if (gi.thr == 0 || gi.valid == 0) continue;
                uint32_t m = 0xFu;   // a threshold of 2^32 selects whatever the word is
                if ((gi.thr >> 32) == 0) {
                    const Philox4 w = philox4x32_10(gi.cgroup, gi.tensor_id, a.step_lo, a.step_hi8, a.keys);
                    const uint32_t thr_lo = static_cast<uint32_t>(gi.thr);
                    m = (w.x < thr_lo ? 1u : 0u) | (w.y < thr_lo ? 2u : 0u) | (w.z < thr_lo ? 4u : 0u) | (w.w < thr_lo ? 8u : 0u);
                }
                sel |= (m & ((1u << gi.valid) - 1u)) << (4 * i);
            }
        }
        if (one_trip) {
            await_previous();
            let_next_start();
            fetch(tile, stage);
            cp_async_wait_all();
        } else cp_async_wait_all_but_latest<1>();   // this tile's copies; the next tile's stay in flight
        __syncwarp();
        if (!__any_sync(0xFFFFFFFFu, sel != 0)) continue;
        const unsigned char *images = smem_raw + stage * stage_bytes;
        const uint32_t count = __reduce_add_sync(0xFFFFFFFFu, __popc(sel));
        const uint32_t thr = (sc.thr_lo >> 1) | (sc.thr_hi << 31);   // half the threshold of the lane's last group
        if (FORM == kServeByCount ? count >= kDenseMinSelected * G : __all_sync(0xFFFFFFFFu, sel == 0 || thr >= a.dense_from) != 0) {
            // every lane serves its own groups, those that are whole; the others go to the list below
#pragma unroll 1
            for (int i = 0; i < G; ++i) {
                const uint32_t mine = (sel >> (4 * i)) & 15u;
                if (!mine) continue;
                const uint32_t g = g_first + i * T_ + lane;
                const GroupInfo gi = find_group_cached(a.pop, sc, g, a.status);
                if (gi.valid != 4) continue;
                sel &= ~(15u << (4 * i));
                const unsigned char *image_a = images + i * (a_bytes + b_bytes);
                if (n_models <= 8) serve_group_dense<TA, TB, LAYOUT, uint32_t>(a, image_a, image_a + a_bytes, g - lane, mine, gi, selected, moved);
                else serve_group_dense<TA, TB, LAYOUT, uint64_t>(a, image_a, image_a + a_bytes, g - lane, mine, gi, selected, moved);
            }
        }
        // the selected coordinates of all G images, 32 at a time, one per lane
        const uint32_t total = list_selected<G>(s_list, sel);
        for (uint32_t first = lane; first < total; first += 32) {
            const uint32_t entry = s_list[first], owner = entry / (4 * G), i = (entry / 4) % G, c = entry & 3u;
            const uint32_t g = g_first + i * T_ + owner;
            uint32_t cgroup = sc.cgroup_begin + (g - sc.begin), tensor = sc.tensor_id;
            if (g - sc.begin >= sc.end - sc.begin) {   // another lane's tensor
                const GroupInfo gi = find_group(a.pop, g, a.status);
                cgroup = gi.cgroup;
                tensor = gi.tensor_id;
            }
            const uint64_t perm = draw_permutation_packed(n_models, 4u * cgroup + c, tensor, a.step_lo, a.step_hi8, a.keys);
            const unsigned char *image_a = images + i * (a_bytes + b_bytes);
            move_coordinate<TA, TB, LAYOUT, FORM == kServeTogether>(a, image_a, image_a + a_bytes, nullptr, perm, owner, c, g - owner, moved);
            ++selected;
        }
        __syncwarp();   // the stage is overwritten by the copies the next trip starts
    }
    cp_async_wait_all();
    publish_warp_stats(a.stats, a.stat_slots, selected, moved);
}

template <class TA, class TB, int G, int kN>
cudaError_t launch_shuffle_loop_tiles(const ShuffleArgs &args, const LaunchShape &shape, cudaStream_t stream)
{
    constexpr bool kHasB = TB::kCode != kDtypeNone;
    const size_t group_elems = 4 * static_cast<size_t>(args.pop.N) + (args.pop.layout == kLayoutPN ? args.pn_pad : 0);
    const size_t image = group_elems * (TA::kBytes + (kHasB ? TB::kBytes : 0)) * 32;
    const size_t smem = (2 * G * image + 2 * 32 * 4 * G + 15) & ~static_cast<size_t>(15);
    const bool np = args.pop.layout == kLayoutNP;
    constexpr int kForm = kN != 0 ? serve_form(kLayoutPN, kN) : kServeByCount;   // (of a population that is compiled in)
    auto kernel = np ? shuffle_loop_kernel<TA, TB, kLayoutNP, G, kN, kServeByCount> : shuffle_loop_kernel<TA, TB, kLayoutPN, G, kN, kForm>;
    if constexpr (kN == 0)
        if (serve_form(args.pop.layout, args.pop.N) == kServeTogether) kernel = shuffle_loop_kernel<TA, TB, kLayoutPN, G, 0, kServeTogether>;
    KernelFit fit;
    cudaError_t err = kernel_fit(reinterpret_cast<const void *>(kernel), 32, smem, &fit);
    if (err != cudaSuccess) return err;
    if (fit.occupancy < 1) return cudaErrorLaunchOutOfResources;
    const uint64_t per_tile = 32ull * G;
    const uint64_t n_tiles = (static_cast<uint64_t>(args.group_hi - args.group_lo) + per_tile - 1) / per_tile;
    if (n_tiles == 0) return cudaSuccess;
    const uint64_t resident = static_cast<uint64_t>(shape.sm_count > 0 ? shape.sm_count : 148) * fit.occupancy;
    return launch_chained(kernel, report_grid(n_tiles, resident), 32, smem, stream, args);
}

template <class TA, class TB>
cudaError_t launch_shuffle_loop_typed(const ShuffleArgs &args, const LaunchShape &shape, cudaStream_t stream)
{
    // Four groups per lane and tile, or two when less than kLoopNarrowShare of the coordinates is expected to
    // be selected: then a trip is short, and more resident warps (32 against 24 on an SM at N = 2) matter more than the
    // serving that four groups share.  Measured (N = 2, fp32, 2^27 coordinates, four / two): p = 1e-4 191 / 176 us, 1e-3
    // 207 / 201, 1e-2 244 / 310; 2^25 coordinates, p = 3e-4 54.1 / 51.5, 1e-3 58.0 / 59.3, 0.1 95.2 / 98.7.  A third stage
    // costs resident warps and was slower everywhere (p = 1e-2 334 us with two groups).
    // (A forced launch may bring groups of any size: beyond kLoopFourMaxGroupBytes four of them leave too few warps.)
    const size_t per_group = static_cast<size_t>(args.pop.N) * 4 * (TA::kBytes + TB::kBytes);
    if (args.expected_share < kLoopNarrowShare || per_group > kLoopFourMaxGroupBytes)
        switch (args.pop.N) {
        case 2: return launch_shuffle_loop_tiles<TA, TB, 2, 2>(args, shape, stream);
        case 3: return launch_shuffle_loop_tiles<TA, TB, 2, 3>(args, shape, stream);
        case 4: return launch_shuffle_loop_tiles<TA, TB, 2, 4>(args, shape, stream);
        case 5: return launch_shuffle_loop_tiles<TA, TB, 2, 5>(args, shape, stream);
        default: return launch_shuffle_loop_tiles<TA, TB, 2, 0>(args, shape, stream);
        }
    switch (args.pop.N) {
    case 2: return launch_shuffle_loop_tiles<TA, TB, 4, 2>(args, shape, stream);
    case 3: return launch_shuffle_loop_tiles<TA, TB, 4, 3>(args, shape, stream);
    case 4: return launch_shuffle_loop_tiles<TA, TB, 4, 4>(args, shape, stream);
    case 5: return launch_shuffle_loop_tiles<TA, TB, 4, 5>(args, shape, stream);
    default: return launch_shuffle_loop_tiles<TA, TB, 4, 0>(args, shape, stream);
    }
}

inline cudaError_t launch_shuffle_loop(const ShuffleArgs &args, int a_dtype, int b_dtype, const LaunchShape &shape,
                                       cudaStream_t stream, bool *supported)
{
    *supported = true;
    if (a_dtype == kDtypeF32 && b_dtype == kDtypeNone) return launch_shuffle_loop_typed<F32, NoStack>(args, shape, stream);
    if (a_dtype == kDtypeBF16 && b_dtype == kDtypeNone) return launch_shuffle_loop_typed<BF16, NoStack>(args, shape, stream);
    if (a_dtype == kDtypeF32 && b_dtype == kDtypeF32) return launch_shuffle_loop_typed<F32, F32>(args, shape, stream);
    if (a_dtype == kDtypeBF16 && b_dtype == kDtypeF32) return launch_shuffle_loop_typed<BF16, F32>(args, shape, stream);
    if (a_dtype == kDtypeBF16 && b_dtype == kDtypeBF16) return launch_shuffle_loop_typed<BF16, BF16>(args, shape, stream);
    if (a_dtype == kDtypeF32 && b_dtype == kDtypeBF16) return launch_shuffle_loop_typed<F32, BF16>(args, shape, stream);
    *supported = false;
    return cudaSuccess;
}

}  // namespace wash
