// Warp tiles: the work unit of the kernels that draw the mask without touching the stacks (the
// sparse shuffle and the one-model-per-device exchange).  A warp tile is 128 consecutive groups
// (512 coordinates); a lane owns four consecutive groups of it, so that its four Philox draws
// overlap, one table lookup serves all four, and its four mask nibbles fit half a word.  A warp
// visits a contiguous range of warp tiles in order.
//
// `A` is the kernel's argument struct; it has the fields pop, keys, step_lo, step_hi8, status.
#pragma once
#include "wash_device.cuh"

namespace wash {

constexpr int kWarpTileGroups = 128;
constexpr uint32_t kFull = 0xFFFFFFFFu;

// The segment a lane's groups were last found in, kept in registers.  While the lane's four
// groups lie among that segment's whole groups a tile costs two compares, four Philox blocks
// and their packing; a tensor's end (its ragged last group, padding) is drawn group by group.
// Starts empty: LaneSegment{}.
struct LaneSegment {
    uint32_t begin = 0, end = 0;     // groups [begin, end) of the row (empty: nothing found yet)
    uint32_t fours = 0;              // from begin + 0 .. fours - 1 on there are four whole groups of it inside the caller's range
    uint32_t cgroup_off = 0;         // group index within the tensor = group + cgroup_off (modulo 2^32)
    uint32_t tensor = 0, thr = 0;    // threshold (0: nothing to draw)
    uint32_t always = 0;             // 0xFFFF when the threshold is 2^32, else 0
};

// Finds group g (inside the row) and loads its segment into the lane's registers; the caller's
// range of groups ends at group_hi.
template <class A>
__device__ __forceinline__ void lane_segment_load(const A &a, uint32_t g, uint32_t group_hi, LaneSegment &ls)
{
    uint32_t s = __ldg(a.pop.tile_first + (g >> kTileShift));
    const uint32_t last = static_cast<uint32_t>(a.pop.n_seg) - 1u;
    uint4 lo = __ldg(reinterpret_cast<const uint4 *>(a.pop.seg + s));       // begin, end, tensor, cgroup_begin
    uint4 hi = __ldg(reinterpret_cast<const uint4 *>(a.pop.seg + s) + 1);   // numel, -, thr
    while (s < last && g >= lo.y) {
        ++s;
        lo = __ldg(reinterpret_cast<const uint4 *>(a.pop.seg + s));
        hi = __ldg(reinterpret_cast<const uint4 *>(a.pop.seg + s) + 1);
    }
    if (g < lo.x || g >= lo.y) {   // table inconsistent with the row: report, select nothing
        if (a.status) atomicOr(a.status, 1u);
        ls = LaneSegment{};
        return;
    }
    ls.begin = lo.x;
    ls.end = lo.y;
    const uint32_t whole = min(hi.x / 4u, group_hi - lo.x);
    ls.fours = whole < 4u ? 0u : whole - 3u;
    ls.cgroup_off = lo.w - lo.x;
    ls.tensor = lo.z;
    ls.thr = hi.z;
    ls.always = hi.w != 0 ? 0xFFFFu : 0u;
}

// The masks of the four consecutive groups from g0 on (bit 4q + c = coordinate c of group g0 + q),
// which are whole groups of the lane's segment.  Four independent chains under one condition, so
// that they interleave.
template <class A>
__device__ __forceinline__ uint32_t draw_four_masks(const A &a, uint32_t g0, const LaneSegment &ls)
{
    if (ls.thr == 0) return ls.always;
    uint32_t w[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const Philox4 block = philox4x32_10(g0 + ls.cgroup_off + q, ls.tensor, a.step_lo, a.step_hi8, a.keys);
        w[4 * q] = block.x;
        w[4 * q + 1] = block.y;
        w[4 * q + 2] = block.z;
        w[4 * q + 3] = block.w;
    }
    return pack_below(w, ls.thr);
}

// the mask of one group: bit c set iff coordinate c is selected
template <class A>
__device__ __forceinline__ uint32_t draw_mask(const GroupInfo &gi, const A &a)
{
    if (gi.thr == 0 || gi.valid == 0) return 0;
    const Philox4 w = philox4x32_10(gi.cgroup, gi.tensor_id, a.step_lo, a.step_hi8, a.keys);
    const uint32_t thr_lo = static_cast<uint32_t>(gi.thr);
    const bool always = (gi.thr >> 32) != 0;
    uint32_t m = 0;
    m |= (w.x < thr_lo || always) ? 1u : 0u;
    m |= (w.y < thr_lo || always) ? 2u : 0u;
    m |= (w.z < thr_lo || always) ? 4u : 0u;
    m |= (w.w < thr_lo || always) ? 8u : 0u;
    return m & ((1u << gi.valid) - 1u);
}

// The masks of groups g0 .. g0+3 of the row, a nibble per group; groups from group_hi on select
// nothing.
template <class A>
__device__ __forceinline__ uint32_t lane_masks(const A &a, uint32_t g0, uint32_t group_hi, LaneSegment &ls)
{
    if (g0 - ls.begin >= ls.fours) {
        if (g0 >= group_hi) return 0;
        if (g0 - ls.begin >= ls.end - ls.begin) lane_segment_load(a, g0, group_hi, ls);
        if (g0 - ls.begin >= ls.fours) {
            uint32_t sel = 0;
#pragma unroll 1
            for (uint32_t q = 0; q < 4 && g0 + q < group_hi; ++q) sel |= draw_mask(find_group(a.pop, g0 + q, a.status), a) << (4 * q);
            return sel;
        }
    }
    return draw_four_masks(a, g0, ls);
}

__device__ __forceinline__ uint32_t warp_exclusive_scan(uint32_t mine, uint32_t *total)
{
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t upto = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t v = __shfl_up_sync(kFull, upto, d);
        if (lane >= static_cast<uint32_t>(d)) upto += v;
    }
    *total = __shfl_sync(kFull, upto, 31);
    return upto - mine;
}

}  // namespace wash
