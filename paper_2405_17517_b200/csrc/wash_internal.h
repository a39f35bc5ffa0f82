// Internal interface between the C ABI (wash_api.cu) and the kernel launchers.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace wash {

constexpr int kMaxN = 64;          // largest population (WASH_MAX_N)
constexpr int kTileShift = 8;      // lookup tile = 256 groups = 1024 coordinates
constexpr int kDtypeF32 = 0, kDtypeBF16 = 1, kDtypeNone = -1;
constexpr int kLayoutNP = 0, kLayoutPN = 1;
constexpr int kModeStream = 0, kModeSparse = 1;

// Values of a selected coordinate that the streaming kernels store with one instruction: neighbouring models' in [P][N]
// (move_neighbours up to 16 models, move_quads above); 1: every value by itself.
__host__ __device__ constexpr int stored_together(int layout, int n_models)
{
    return layout != kLayoutPN || n_models == 2 ? 1 : n_models % 4 == 0 ? 4 : n_models % 2 == 0 && n_models <= 16 ? 2 : 1;
}

// How a streaming kernel serves what a warp has selected.  The forms are kernels of their own: the code of one costs the populations
// of another up to 12 % (N = 7 bf16, p = 0.4 176 us alone, 198 with the code that stores values together; 4 % by the choice at run time).
//   kServeByCount      values one by one, densely from half of a warp's coordinates on: [N][P], odd populations, more than 16 models
//   kServeByThreshold  values one by one, densely from a threshold on (dense_threshold): two models in [P][N]
//   kServeTogether     neighbouring models' values together, densely from a threshold on: even populations from 4 to 16 models in [P][N]
constexpr int kServeByCount = 0, kServeByThreshold = 1, kServeTogether = 2;
__host__ __device__ constexpr int serve_form(int layout, int n_models)
{
    return layout != kLayoutPN || n_models > 16 ? kServeByCount : n_models == 2 ? kServeByThreshold : stored_together(layout, n_models) > 1 ? kServeTogether : kServeByCount;
}

// One row of a stack is cut into groups of 4 consecutive elements; a group never
// straddles two tensors because tensors start on multiples of 8 elements.
struct SegEntry {
    uint32_t group_begin;   // first group of the segment within a row
    uint32_t group_end;     // one past its last group (padding groups included)
    uint32_t tensor_id;     // RNG tensor index
    uint32_t cgroup_begin;  // (first coordinate's index within its tensor) / 4
    uint32_t numel;         // coordinates in the segment
    uint32_t reserved;
    uint64_t thr;           // floor(p * 2^32): coordinate selected iff word < thr
};
static_assert(sizeof(SegEntry) == 32, "SegEntry must stay 32 bytes");

// Statistics are gathered in kStatSlots partial sums before they reach the caller's two
// counters: per-block atomics on one address were measured to cost about 1 ns each and
// to dominate the kernel once most blocks have a selected coordinate.  One more slot gathers the sums of a launch whose
// counters lie in host memory.
constexpr int kStatSlots = 256;
struct StatSlot {
    unsigned long long selected, moved;
    unsigned long long report;   // resident-warp streaming kernel: blocks that have reported and their counters (publish_warp_stats)
    unsigned long long reserved;
};

struct PopView {
    int N;
    int layout;
    long long padded_P;           // elements per model row
    uint32_t n_groups;            // padded_P / 4
    int n_seg;
    const SegEntry *seg;          // device, n_seg entries
    const uint32_t *tile_first;   // device, segment of the first group of every tile
};

// Philox's key schedule: round r of the ten uses (k[2r], k[2r+1]) = (seed_lo + r W0, seed_hi + r W1)
// with the two Weyl constants.  It depends on the seed only, so the host computes it once per
// launch and a round's key reaches the kernel as an operand instead of two additions.
struct PhiloxKeys {
    uint32_t k[20];
};
inline PhiloxKeys philox_keys(uint64_t seed)
{
    PhiloxKeys keys;
    uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
    for (int r = 0; r < 10; ++r, k0 += 0x9E3779B9u, k1 += 0xBB67AE85u) {
        keys.k[2 * r] = k0;
        keys.k[2 * r + 1] = k1;
    }
    return keys;
}

// Distance to the consensus gathered inside the streaming shuffle: up to kMaxSqRanges ranges of
// segments, per range and model a binary64 sum, gathered in kSqSlots partial copies (atomics on
// one address per model would serialise) that sq_flush_kernel adds into the caller's array.
constexpr int kMaxSqRanges = 8;
constexpr int kSqSlots = 64;
struct SqArgs {
    double *slots = nullptr;                // device: [kSqSlots][n_ranges][N], zero between launches; nullptr = statistic off
    int n_ranges = 0;
    double inv_n = 0.0;                     // 1 / N
    uint32_t seg_bound[kMaxSqRanges + 1];   // range r = segments seg_bound[r] .. seg_bound[r+1]-1
};

struct ShuffleArgs {
    PopView pop;
    void *a;                      // first stack (device)
    void *b;                      // second stack or nullptr
    uint32_t group_lo, group_hi;  // groups of a row to process (whole row: 0 .. n_groups)
    PhiloxKeys keys;              // from the seed
    uint32_t step_lo, step_hi8;   // step & 0xFFFFFFFF, (step >> 32) << 8
    unsigned long long *stats;    // device-accessible {selected, moved} or nullptr
    StatSlot *stat_slots;         // device, kStatSlots + 1 zeroed entries (left zeroed by every launch)
    bool stats_direct = false;    // few blocks report: they add to `stats` themselves (kernels that need a flush kernel otherwise)
    uint32_t dense_from = 0xFFFFFFFFu;   // streaming kernels, even populations of up to 16 models in [P][N]: half the threshold from which a tensor is served densely (dense_threshold)
    uint32_t *status;             // device status word
    SqArgs sq;                    // consensus distance of the first stack (streaming kernel only)
    bool measure_only = false;    // with sq: nothing is selected
    uint32_t pn_pad = 0;          // streaming kernel, [P][N]: elements of padding after a group in the shared-memory image (0 or 4)
    uint32_t pair_inverse = 0;    // streaming kernel, N > 16: 2^20 / N, rounded up (i / N = i * pair_inverse >> 20 for i < 2^14, and i is at most 64 N; set by its launcher)
    bool early = false;           // streaming kernel: the flavour that draws permutations while the copies are in flight
    void *mirror_a = nullptr;     // sparse kernel: a second copy of each stack (mapped host memory) that receives the moved values, too
    void *mirror_b = nullptr;
    float expected_share = 0.f;   // share of the coordinates the call's probabilities select, in expectation (sizes the sparse kernel's grid)
};
// A launch with more than 288 bytes of arguments costs the host 0.35 us more (3.4 -> 3.75 us a call with 296).
static_assert(sizeof(ShuffleArgs) <= 288, "ShuffleArgs must stay within 288 bytes");

// Whether the sparse kernels' loads of values ask for 64 bytes of a line instead of all 128 (load_scattered).  128 bytes are the better
// request where a line's other half holds a selected coordinate as well, which is then fetched for nothing, and where masks and not
// values are most of the time the two are alike and the plain load costs fewer instructions.  Time with 64 bytes over time with 128, stacks of 400 MB:
//   [N][P], 1 / 2 / 4 / 6 % selected (10 %): fp32 N = 3 1.01 1.00 .98 .97 (1.01), 5 .98 .93 .92 .96 (1.07), 8 .97 .93 .96 1.01, 16 .98 .97 1.01 1.07, 24 1.00 1.02
//     1.09, 48 .99 1.04, 64 1.03 1.05;  bf16 8 .98 .95 1.06 1.16, 16 .96 .99 1.12, 24 1.00 1.07, 48 1.03 1.16;  two fp32 stacks 2 1.02 1.02 .92 .88 (.91), 3 .99 .92 .90 .92 (.99), 8 1.00 .98
//     .99 1.02, 24 .97 .99 1.08;  bf16 + fp32, in either order 3 1.00 .93 .90 .96 (1.05), 5 .96 .94 .97 1.02, 8 .98 .98 1.01 1.06, 12 1.00 .99 1.03, 24 .98 1.02 1.10, 32 .98 1.02
//     1.12;  by warps (shuffle_sparse_warps_kernel), 6 / 10 % fp32 24 .92 .95, 64 .94 .97, bf16 24 .97 .99, bf16 + fp32 .94 .96.
//     Few values, .002 to .003 of a coordinate's: 1.00 to 1.03 up to .03 values a coordinate (N = 5 two stacks, p = 2e-3 1.03), from .04 on .97 to 1.00.
//   [P][N], one stack: 1.00 to 1.03 throughout.  Two stacks, 1 / 2 / 4 / 6 / 10 %: fp32 N = 3 1.01 .98 .93 .90 .93, 5 1.00 .99 .97 .95 .90, 8 1.00 1.01 .98 .96 .94, 12 1.01 1.02 .99
//     .98 .99, 16 1.00 1.02 1.03 1.02 1.02, 32 1.01 1.02 1.01; bf16 + fp32 3 1.00 .99 .95 .91 .98, 5 1.01 .98 .95 .92 .94, 24 1.00 1.01 1.02 1.02 1.03.
// ResNet-50 N = 8, bf16 + fp32, p = 5e-3: 77.2 -> 71.3 us, N = 5, p = 0.05 -> 0 46.8 -> 44.9.
inline bool fetch_half_lines(const ShuffleArgs &args, bool by_warps, int bytes_a, int bytes_b)
{
    const int N = args.pop.N;
    const bool two_stacks = bytes_b != 0;
    const float elem = two_stacks ? 0.5f * static_cast<float>(bytes_a + bytes_b) : static_cast<float>(bytes_a);   // the stacks are asked alike
    const float values = args.expected_share * static_cast<float>(N), per_line = args.expected_share * 128.f / elem;
    if (args.pop.layout == kLayoutPN) return two_stacks && N <= 12 && values >= 0.06f && per_line < static_cast<float>(N);
    return values >= 0.035f && per_line < (by_warps ? 4.f : N <= 3 ? 3.f : N <= 5 ? 2.f : N <= 16 ? 1.5f : N <= 32 ? 0.7f : 0.f);
}

// Whether half a wave of blocks serves a sparse launch of `n_wtiles` warp tiles whose values would be `by_load` blocks' (launch_shuffle_sparse_typed
// has the units).  Launches that follow each other at once gain by it: a launch's masks are drawn beside the serving of the one before, which a
// whole wave leaves no room, and 16 warps draw masks at nearly the rate of 32.  A launch behind a kernel that releases nothing early, an
// optimizer's in a training loop, gains nothing and waits for blocks that serve twice as much.  us, whole -> half: call after call | behind an elementwise
// kernel on other data | behind one on the stacks (chains less the chains without the shuffle):
//   ResNet-18 N = 5, p = 3e-4 10.2 -> 9.1 | 12.5 -> 12.4 | 13.5 -> 13.4;  with momentum, p = 1e-3 (0.32 of a wave) 10.9 -> 9.5 | 14.3 -> 16.1 | 14.1 -> 14.8
//   N = 2, 2^23 coordinates, p = 1e-3 8.0 -> 7.2 | 10.2 -> 10.2 | 10.2 -> 10.2;  N = 10, 2^23, 5e-4 8.9 -> 7.4 | 10.5 -> 10.6 | 11.2 -> 11.2;  N = 16 bf16, 2^23, 5e-4 9.3 ->
//   7.6 | 12.3 -> 12.3 | 14.0 -> 14.2;  N = 5, 2^24, 1e-3 14.2 -> 13.5 | 18.4 -> 18.4 | 18.0 -> 18.3;  [P][N] N = 8, 2^24, 1e-3 13.9 -> 13.1 | 16.5 -> 17.1 | 17.6 -> 17.8
// So ResNet-18 with momentum, 0.32 of a wave, loses behind other kernels up to what it gains; from 0.4 on more, as rows of more than 16 tiles a warp do, and
// populations of 48 models, whose coordinate is a block's work for a while, lose both ways (N = 20, 2^22, 1e-3 6.9 -> 6.6 | 10.2 -> 10.3 | 9.6 -> 9.6):
//   N = 5 with momentum, 2^24, 1e-3 (0.47) 14.3 -> 13.4 | 20.3 -> 22.4 | 18.7 -> 20.9;  N = 3, 2^25, 3e-4 (28 tiles) 25.1 -> 24.4 | 28.7 -> 30.2 | 29.2 -> 30.3
//   N = 48, 2^21, 1e-3 8.0 -> 8.4 | 10.7 -> 12.1 | 9.7 -> 10.5;  [P][N], 3e-3 6.8 -> 7.2 | 8.2 -> 8.3 | 8.0 -> 8.9
// Five eighths to seven eighths of a wave gain less and lose as much (ResNet-18 with momentum 0.75: 11.4 | 14.3 | 14.2).  Waves and a half lose (N = 3 two
// stacks, p = 5e-3, 1.5 waves 20.7, two 18.9).
// More than 32 models with few values a block gain, call after call: N = 64 bf16, 3e-4 (100 values) [N][P] 7.8 -> 7.3, [P][N] 6.8 -> 5.9; [P][N], whose values are neighbours,
// 1e-3 (340) 7.7 -> 6.9; N = 48 above has 170 in [N][P] and 510 in [P][N].  `expected` coordinates in `stacks` stacks.
inline bool half_wave_serves(int layout, int n_models, int stacks, double expected, double by_load, uint32_t resident, uint32_t n_wtiles)
{
    const double values = expected * n_models * stacks / (0.5 * resident);   // of a block
    if (n_models > 32 && values > (layout == kLayoutNP ? 128.0 : 400.0)) return false;
    return by_load <= 0.4 * resident && n_wtiles <= 32ull * resident;   // 16 tiles for each of the 4 warps of resident / 2 blocks
}

// [P][N], even populations of up to 16 models: the threshold from which every lane serves its own group (serve_group_dense) instead of
// coordinates dealt to the lanes, whose values are stored together from 4 models on.  It is the tensor's threshold that decides, not what a
// warp happens to have selected: warps of both kinds beside each other take longer than those of either (N = 2 fp32, 2^24 coordinates, p = 0.8, from 100 selected of
// a warp's 128 on 165 us, all dense 130, all dealt 161; two fp32 stacks 278, 212, 262).  Time dense over time dealt at 45 / 55 / 65 / 75 / 80 / 85 / 90 / 100 %:
//   one stack   fp32 N = 2 1.19 1.00 .97 .87 .81 .80 .80 .80, 4 1.43 1.20 1.16 1.04 .96 .95 .95 .96, 6 1.42 1.16 1.12 1.00 .93 .91 .91 .90, 8 2.40 1.20 1.15 1.03 .98 .96 .96 .96, 10
//               1.59 1.29 1.25 1.10 1.01 1.00 1.00 1.00, 12 1.65 1.33 1.29 1.13 1.04 1.04 1.03 1.04, 14 as 10, 16 2.81 1.36 1.33 1.18 1.10 1.08 1.07 1.07;  bf16 2 1.20 1.00 .97
//               .88 .82 .81 .81 .80, 4 1.36 1.14 1.10 .99 .92 .91 .91 .91, 8 1.61 1.31 1.25 1.10 1.00 .98 .98 .98, 10 to 16 as fp32
//   two stacks  fp32 N = 2 1.15 .98 .95 .86 .80 .79 .79 .77, 4 1.99 1.14 1.22 1.11 1.10 1.08 1.07 1.14, 6 1.27 1.17 1.11 .99 1.00 .99 .93 .94, 8 3.20 1.96 1.92 1.78 1.71 1.66 1.65 1.58, 10 1.56 1.42
//               1.28 1.16 1.13 1.08 1.02 .92, 12 2.40 1.81 1.79 1.65 1.62 1.57 1.51 1.51, 14 1.61 1.47 1.33 1.18 1.12 1.07 1.02 .95, 16 3.16 2.01 1.98 1.87 1.78 1.75 1.72 1.59;  bf16 + fp32 4 1.86 1.12 1.13
//               1.02 .95 .93 .94 .94, 6 1.30 1.12 1.21 1.02 .99 1.00 .98 .97, 8 to 16 by fours 1.3 to 3.6, 10 1.22 1.24 1.14 1.07 1.04 1.03 .99 .95, 14 1.34 1.24 1.13 1.02 .99 .96 .92 .86
inline uint32_t dense_threshold(int n_models, bool two_stacks, bool all_f32)   // (half of it: it may be 2^32)
{
    const float share = n_models == 2 ? 0.56f : n_models <= 8 ? 0.78f : !two_stacks ? 0.85f : all_f32 ? 0.88f : 0.79f;
    if (n_models % 4 == 0 && (two_stacks ? n_models > 4 || all_f32 : n_models > 8)) return 0xFFFFFFFFu;   // never
    return static_cast<uint32_t>(share * 2147483648.f);
}

// Blocks of the resident-warp streaming kernel: those that are resident, as far as there are tiles for them -- and, where a device has few
// SMs, so many that the counters of a slot fit the fields they are reported in (publish_warp_stats): fewer than 256 blocks and fewer than
// 2^26 selected coordinates to a slot.  A row has fewer than 2^33 coordinates; one slot in kStatSlots gets ceil(grid / kStatSlots) of the grid's equal
// shares, which is at most 2 / 257 of the row for a grid of kStatSlots blocks or more and could be all of it for smaller ones.
inline uint32_t report_grid(uint64_t n_tiles, uint64_t resident)
{
    constexpr uint64_t kLeast = kStatSlots, kMost = 255ull * kStatSlots;
    const uint64_t grid = resident < kLeast ? kLeast : resident > kMost ? kMost : resident;
    return static_cast<uint32_t>(n_tiles < grid ? n_tiles : grid);
}

// Whether the blocks of shuffle_wide_pn_kernel fetch their bytes by bulk copies.  Only where a wait that is given up can be reported: without a
// status word (wash_shuffle_noalloc) the block would stay as it was, and nobody would know.  A bulk copy takes multiples of 16 bytes: groups come
// in pairs (rows and ranges are whole units of 8 elements) and have 8 N bytes at least.
// Time with bulk copies over time with 16 bytes (bf16: 8) a thread at a time, by bytes of a block's images (32 groups, 64 for N <= 39 in fp32 and like sizes), 1 / 3 /
// 10 / 30 % selected, stacks of 0.4 GB, and of 3 GB:
//   one stack    fp32  22 KB (N = 44) .92 .84 .85 .90, 1.34 1.41 .85 .90;  25 KB (48) .94 .85 .84 .90, 1.30 1.24 .85 .90;  27 KB (52) .91 .83 .84 .90, 1.18 .83 .84 .90;  29 KB (56) .93 .84
//                .84 .90, 1.13 1.21 .84 .90;  30 KB (58 to 60) .88 .82 .85, .88 .82 .85;  33 KB (32, 64) .95 .91 .88 .90, .97 .92 .87 .90;  37 KB (36) .91 .87 .86 .90, the same
//   two stacks   bf16 + fp32  22 KB (28) .93 .87 .89 .85, 1.42 1.55 1.33 .84;  25 KB (32) .91 .85 .83 .84, 1.27 1.40 .87 .83;  28 KB (36) .89 .82 .83 .84, 1.12 1.26 .84 .83;  31 KB (40) .85 .77 .77
//                .84, .89 1.09 .96 .83;  32 to 34 KB (42 to 44, 22) .86 .78 .79 .84, .88 .79 to 1.03 .79 .83;  37 KB (24, 48) .85 .80 .82 .85, .86 .82 .82 .84
//                fp32 twice  25 KB (24) .96 .94 .96 .87, 1.33 1.61 1.42 .87;  33 KB (32) .95 .89 .86 .85, .99 1.22 1.00 .85;  34 and 35 KB (33, 34; 17) .96 .90 .86 .84, .99 1.16 .88 .85;  35 KB and
//                more of 32 groups (35, 36) .93 .84 .82 .85, .95 .84 to 1.04 .84 .85;  37 to 41 KB of 64 groups (18, 20) .96 .95 .94 .89, .99 to 1.18 1.12 .95 .88;  49 and 65 KB (48, 64) .86 .76 .76 .84, the same
//                bf16 twice  20 KB (40) .68 .71 .75, 1.15 1.20 .69 .73;  25 KB (48) .70 .65 .68 .80, .95 .65 to 1.03 .67 .80;  33 KB (32, 64) .68 .65 .68 .80, the same
// So they pay where much is selected, for large blocks, and in stacks of up to half a GB (400 MB: .63 to 1.00 in all of 420 cells); small blocks of
// which little is selected lose in stacks of 0.8 to 1.6 GB and more, for a reason that is not known.  N = 32 fp32, 2^25 coordinates, p = 0.1 813 -> 707 us.
inline bool copies_in_bulk(const ShuffleArgs &args, uint32_t groups, int bytes_a, int bytes_b)
{
    if (!args.status || args.pn_pad != 0 || ((args.group_lo | args.group_hi) & 1u) != 0) return false;
    const uint32_t group_bytes = 4u * static_cast<uint32_t>(args.pop.N * (bytes_a + bytes_b)), image = groups * group_bytes;
    const float share = args.expected_share;
    if (static_cast<uint64_t>(args.group_hi - args.group_lo) * group_bytes <= 500000000u) return true;
    if (bytes_a != 4 && bytes_b != 4) return share >= 0.08f || image >= 24000u;
    if (share >= 0.2f) return true;
    if (bytes_b == 0) return image >= 29500u;
    if (bytes_a != bytes_b) return image >= 32000u;
    return share >= 0.08f ? image >= 33000u : group_bytes >= 1120u;
}

struct ReduceArgs {
    PopView pop;
    void *stack;                  // device stack (read; written by EMA / papa_all)
    void *out;                    // average row (device) or nullptr
    float alpha, one_minus_alpha;
    uint32_t group_lo, group_hi;  // range of groups to process (both even: whole units of 8 elements)
    uint32_t *status;
};

// One model per device (wash_exchange_*): the row is one model of a population of pop.N.
constexpr int kExchangeTileGroups = 128;   // a warp tile (wash_warp_tiles.cuh): 32 lanes x 4 groups = 512 coordinates
constexpr int kExchangeWarps = 8;          // warps per block of the exchange kernels
constexpr int kExchangeBlocksPerSm = 4;    // resident blocks of the plan kernel on an SM
struct ExchangeArgs {
    PopView pop;
    int self;                     // this worker's index in the population
    uint32_t n_wtiles;            // ceil(n_groups / kExchangeTileGroups)
    uint32_t n_blocks;            // grid of all three kernels; its blocks share the warp tiles evenly, in order
    PhiloxKeys keys;
    uint32_t step_lo, step_hi8;
    uint32_t *mask;               // [n_wtiles * 32] a word per lane, a nibble per group; low half:
                                  // selected coordinates, high half: those this worker receives
    uint32_t *block_total;        // [n_blocks][N + 1]: column n = slots of worker n's buffer the block's range takes; column N = selected coordinates
    void *row[2];                 // this worker's model: parameters, optimizer state (nullptr: absent)
    int dtype[2];
    void *const *staging[2];      // per stack: device array of N pointers, entry n = worker n's staging buffer
    long long capacity[2];        // elements per staging buffer
    unsigned long long *stats;    // {selected, received} or nullptr
    uint32_t *status;
};
cudaError_t launch_exchange_plan(const ExchangeArgs &args, cudaStream_t stream);
cudaError_t launch_exchange_send(const ExchangeArgs &args, cudaStream_t stream);
cudaError_t launch_exchange_receive(const ExchangeArgs &args, cudaStream_t stream);

enum ReduceOp { kOpEma = 0, kOpAverage = 1, kOpPapaAll = 2 };

// The resident-warp streaming kernel takes groups (all models, both stacks) of up to 48 bytes -- fp32 N = 2, 3;
// bf16 N <= 6 -- when at most 30 % of the coordinates are expected to be selected, and two groups per lane instead of four
// below kLoopNarrowShare (see its launcher).  Against the one-trip kernel, 2^25 coordinates: 32 bytes 0.6-0.9 of its time.
constexpr size_t kLoopMaxGroupBytes = 48;
constexpr size_t kLoopFourMaxGroupBytes = 128;
constexpr float kLoopMaxShare = 0.3f, kLoopNarrowShare = 0.0007f;
// N > 16: below this expected selection the one-trip kernel's own serving (a single coordinate of a warp served by the
// whole warp) is as good (N = 20 .. 64, p = 1e-3: 0.97-1.03 of the wide kernel's time; N = 17 in bf16 26.6 against 27.6 us for
// 4.0 M coordinates); at 1 % the wide kernel takes 0.65-0.99 of its time.
constexpr float kWideMinShare = 0.003f;

struct LaunchShape {
    int threads;         // 0 = default
    int blocks_per_sm;   // streaming shuffle: which kernel (wash_set_launch)
    int sm_count;
};

// Each returns cudaSuccess or the launch error; *supported = false (and no launch) if
// the library has no kernel for the combination.
cudaError_t launch_shuffle(const ShuffleArgs &args, int a_dtype, int b_dtype, int mode,
                           const LaunchShape &shape, cudaStream_t stream, bool *supported);
cudaError_t launch_reduce(const ReduceArgs &args, int op, int dtype, int out_dtype,
                          const LaunchShape &shape, cudaStream_t stream, bool *supported);

// adds the slots' sums into out[n_ranges][N] and zeroes the slots
cudaError_t launch_sq_flush(const SqArgs &sq, int N, double *out, cudaStream_t stream);

cudaError_t launch_philox_probe(unsigned long long n_blocks, uint64_t seed, uint32_t *checksum, cudaStream_t stream);

void count_launch();

}  // namespace wash
