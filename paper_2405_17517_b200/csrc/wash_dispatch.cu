// Chooses the shuffle kernel of a call, and the small kernels beside them.
#include <atomic>
#include "wash_internal.h"
#include "wash_device.cuh"
#include "wash_launch.cuh"

namespace wash {

cudaError_t launch_reduce_f32(const ReduceArgs &, int, int, const LaunchShape &, cudaStream_t);
cudaError_t launch_reduce_bf16(const ReduceArgs &, int, int, const LaunchShape &, cudaStream_t);
cudaError_t launch_shuffle_sparse(const ShuffleArgs &, int, int, const LaunchShape &, cudaStream_t, bool *);
cudaError_t launch_shuffle_stream(const ShuffleArgs &, int, int, const LaunchShape &, cudaStream_t, bool *);
cudaError_t launch_shuffle_stream_wide(const ShuffleArgs &, int, int, const LaunchShape &, cudaStream_t, bool *);
cudaError_t launch_shuffle_stream_loop(const ShuffleArgs &, int, int, const LaunchShape &, cudaStream_t, bool *);

static std::atomic<uint64_t> g_launches{0};
void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
uint64_t launch_count() { return g_launches.load(std::memory_order_relaxed); }

// Sums the partial statistics into the caller's counters and zeroes them again.
// (Warp shuffles, then eight partial sums: 64-bit atomics on one shared-memory word are
// compare-and-swap loops and cost this one-block kernel 20 us when 256 threads contended.)
__global__ void __launch_bounds__(kStatSlots) flush_stats_kernel(StatSlot *slots, unsigned long long *stats)
{
    await_previous();
    let_next_start();
    __shared__ unsigned long long part[2][kStatSlots / 32];
    unsigned long long sel = slots[threadIdx.x].selected, mov = slots[threadIdx.x].moved;
    if (sel) {
        slots[threadIdx.x].selected = 0;
        slots[threadIdx.x].moved = 0;
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        sel += __shfl_down_sync(0xFFFFFFFFu, sel, d);
        mov += __shfl_down_sync(0xFFFFFFFFu, mov, d);
    }
    if ((threadIdx.x & 31) == 0) {
        part[0][threadIdx.x >> 5] = sel;
        part[1][threadIdx.x >> 5] = mov;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long s = 0, m = 0;
#pragma unroll
        for (int w = 0; w < kStatSlots / 32; ++w) {
            s += part[0][w];
            m += part[1][w];
        }
        if (s) {
            atomicAdd(stats, s);
            atomicAdd(stats + 1, m);
        }
    }
}

// Adds a launch's two counters, gathered on the device, to the caller's in host memory and zeroes them again.
__global__ void __launch_bounds__(32) hand_over_stats_kernel(StatSlot *total, unsigned long long *stats)
{
    await_previous();
    let_next_start();
    if (threadIdx.x != 0 || total->selected == 0) return;
    atomicAdd(stats, total->selected);
    atomicAdd(stats + 1, total->moved);
    total->selected = 0;
    total->moved = 0;
}

// Adds the kSqSlots partial copies of the [range][model] table of squared distances into the
// caller's array and leaves the slots zeroed for the next launch.  A warp per entry, a lane per two
// copies (a thread that went through the copies of an entry one after the other took 64 round trips).
__global__ void __launch_bounds__(1024) sq_flush_kernel(double *slots, int count, double *out)
{
    await_previous();
    let_next_start();
    static_assert(kSqSlots == 64, "two copies per lane");
    const int lane = threadIdx.x & 31;
    for (int j = threadIdx.x >> 5; j < count; j += blockDim.x >> 5) {
        double *lo = slots + lane * count + j, *hi = lo + 32 * count;
        double s = *lo + *hi;
        *lo = 0.0;
        *hi = 0.0;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xFFFFFFFFu, s, d);
        if (lane == 0) atomicAdd(out + j, s);   // contexts on other streams may add to the same array
    }
}

cudaError_t launch_sq_flush(const SqArgs &sq, int N, double *out, cudaStream_t stream)
{
    const int entries = sq.n_ranges * N;
    return launch_chained(sq_flush_kernel, 1, entries < 32 ? 32 * entries : 1024, 0, stream, sq.slots, entries, out);
}

// Nothing but the mask's Philox blocks: four blocks per thread (four independent chains, as in the
// kernels that draw masks without touching memory), folded by XOR.  With one block per thread the
// same kernel measures a quarter less (3.17 against 4.2e11 blocks/s): the chains' latency shows.
__global__ void __launch_bounds__(256) philox_probe_kernel(unsigned long long n_blocks, const __grid_constant__ PhiloxKeys keys, uint32_t *checksum)
{
    const unsigned long long i = (static_cast<unsigned long long>(blockIdx.x) * blockDim.x + threadIdx.x) * 4ull;
    uint32_t fold = 0;
    if (i + 3 < n_blocks) {   // the four chains under one condition, so that they interleave
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const Philox4 w = philox4x32_10(static_cast<uint32_t>(i + q), 0u, 0u, static_cast<uint32_t>((i + q) >> 32) << 8, keys);
            fold ^= w.x ^ w.y ^ w.z ^ w.w;
        }
    } else {
        for (int q = 0; q < 4 && i + q < n_blocks; ++q) {
            const Philox4 w = philox4x32_10(static_cast<uint32_t>(i + q), 0u, 0u, static_cast<uint32_t>((i + q) >> 32) << 8, keys);
            fold ^= w.x ^ w.y ^ w.z ^ w.w;
        }
    }
    fold = __reduce_xor_sync(0xFFFFFFFFu, fold);
    if (checksum && (threadIdx.x & 31) == 0 && fold == 0x9E3779B9u) atomicAdd(checksum, 1u);   // keeps the work alive; rarely true
}

cudaError_t launch_philox_probe(unsigned long long n_blocks, uint64_t seed, uint32_t *checksum, cudaStream_t stream)
{
    if (n_blocks == 0) return cudaSuccess;
    const unsigned long long grid = ((n_blocks + 3) / 4 + 255) / 256;
    if (grid > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    philox_probe_kernel<<<static_cast<unsigned>(grid), 256, 0, stream>>>(n_blocks, philox_keys(seed), checksum);
    count_launch();
    return cudaGetLastError();
}

// Whether the resident-warp kernel takes a launch whose groups have `per_group` bytes over all models.  It does up
// to kLoopMaxGroupBytes while at most kLoopMaxShare is expected to be selected; larger groups only where serving, which it
// does once per four groups of a lane, weighs most against its fewer resident warps.  Its time over the one-trip
// kernel's, 2^24 coordinates, at 0.3 / 0.5 / 1 / 2 / 5 / 8 / 12 %:
//   32-48     bf16 [P][N], whose values are picked out of the image two bytes at a time: N = 4 at 15 / 20 / 30 % .91 1.08 1.09, N = 5 at
//             10 / 13 / 20 / 30 % .82 .99 1.27 1.29, N = 6 .96 1.11 1.43 1.44
//   64 bytes  fp32 N = 4  [N][P] .97 .89 .81 .83 .94 1.01 1.06   [P][N] .97 .87 .72 .66 .75 .87 .94   (two stacks of N = 2 alike)
//             bf16 N = 8  [N][P] .94 .80 .65 .70 .76 .77 .87     [P][N] .97 .89 .78 .71 .91 1.11 1.23
//   80        fp32 N = 5  [N][P] .89 .90 .89 .91 1.01 1.09 1.16  [P][N] .88 .87 .78 .73 .80 .92 1.05
//             bf16 N = 10 [N][P] 1.08 .98 .80 .81 .81 .81 .95    [P][N] 1.20 1.08 .88 .74 .85 1.06 1.19
//   96        bf16 N = 12 [N][P] 1.18 1.04 .85 .86 .85 .88 1.03  [P][N] 1.30 1.17 .97 .90 1.07 1.28 1.28
//             two fp32 stacks of N = 3 [N][P] 1.01 1.02 1.02 1.07 1.10 1.14 1.19  [P][N] 1.03 .99 .90 .90 1.07 1.15 1.19
//   128       fp32 N = 8  [P][N] 1.15 1.12 .97 .82 .92 1.05 1.21
static bool resident_warps_pay(size_t per_group, int layout, bool bf16, bool two_stacks, float share)
{
    const bool np = layout == kLayoutNP, one_bf16 = bf16 && !two_stacks;
    if (per_group <= kLoopMaxGroupBytes) return share <= (one_bf16 && !np && per_group >= 32 ? 5.2f / per_group : kLoopMaxShare);
    if (per_group <= 64) return share >= 0.003f && share <= (one_bf16 ? (np ? 0.12f : 0.06f) : (np ? 0.07f : 0.12f));
    if (per_group > 96) return false;
    if (two_stacks) return !np && share >= 0.008f && share <= 0.03f;
    if (bf16) return np ? share >= 0.008f && share <= 0.1f : share >= 0.01f && share <= 0.04f;
    return np ? share >= 0.004f && share <= 0.025f : share >= 0.006f && share <= 0.08f;
}

// *flush: the kernel leaves its counters in the partial-sum slots
static cudaError_t launch_shuffle_kernel(const ShuffleArgs &args, int a_dtype, int b_dtype, int mode,
                                         const LaunchShape &shape, cudaStream_t stream, bool *supported, bool *flush)
{
    *flush = args.stats && !args.stats_direct;
    if (mode == kModeSparse) return launch_shuffle_sparse(args, a_dtype, b_dtype, shape, stream, supported);
    // Three streaming kernels.  Small groups of all models (both stacks) go to the resident-warp kernel, whose
    // instruction count per group is a fraction of the one-trip kernel's (resident_warps_pay); larger
    // groups, the consensus statistic and the early flavour stay with the one-trip kernel; populations of more
    // than 16 models have a one-trip kernel of their own from kWideMinShare on, until the early flavour takes over
    // (in [P][N] with a multiple of four models it does not).
    // blocks_per_sm of wash_set_launch: -4 forces the resident-warp kernel, -5 the one-trip kernel.
    const size_t elem_a = a_dtype == kDtypeF32 ? 4 : a_dtype == kDtypeBF16 ? 2 : 0, elem_b = b_dtype == kDtypeF32 ? 4 : b_dtype == kDtypeBF16 ? 2 : 0;
    const size_t per_group = static_cast<size_t>(args.pop.N) * 4 * (elem_a + elem_b);
    bool loop = resident_warps_pay(per_group, args.pop.layout, a_dtype == kDtypeBF16, b_dtype != kDtypeNone, args.expected_share);
    if (shape.blocks_per_sm == -4) loop = true;
    if (shape.blocks_per_sm == -5 || args.sq.slots || args.early || args.pop.N > 16) loop = false;
    if (loop) {
        *flush = false;
        return launch_shuffle_stream_loop(args, a_dtype, b_dtype, shape, stream, supported);
    }
    if (args.pop.N > 16 && !args.early && args.expected_share >= kWideMinShare) return launch_shuffle_stream_wide(args, a_dtype, b_dtype, shape, stream, supported);
    return launch_shuffle_stream(args, a_dtype, b_dtype, shape, stream, supported);
}

cudaError_t launch_shuffle(const ShuffleArgs &args, int a_dtype, int b_dtype, int mode,
                           const LaunchShape &shape, cudaStream_t stream, bool *supported)
{
    // Counters in host memory: an atomic crosses PCIe and takes about a microsecond, one after the other, and a launch has
    // hundreds of blocks that report (2^20 coordinates, N = 3: 437 us, 16 us with counters on the device; sparse 949 us).  Such a
    // launch counts into the spare slot on the device, and one more kernel hands the two sums over.
    ShuffleArgs call = args;
    call.dense_from = dense_threshold(args.pop.N, b_dtype != kDtypeNone, a_dtype == kDtypeF32 && b_dtype != kDtypeBF16);
    cudaPointerAttributes where;
    bool hand_over = false;
    if (args.stats) {
        if (cudaPointerGetAttributes(&where, args.stats) != cudaSuccess) cudaGetLastError();
        else hand_over = where.type != cudaMemoryTypeDevice;
        if (hand_over) call.stats = &args.stat_slots[kStatSlots].selected;   // {selected, moved}
    }
    bool flush = false;
    cudaError_t err = launch_shuffle_kernel(call, a_dtype, b_dtype, mode, shape, stream, supported, &flush);
    if (err != cudaSuccess || !*supported) return err;
    if (flush && (err = launch_chained(flush_stats_kernel, 1, kStatSlots, 0, stream, call.stat_slots, call.stats)) != cudaSuccess) return err;
    if (hand_over) err = launch_chained(hand_over_stats_kernel, 1, 32, 0, stream, call.stat_slots + kStatSlots, args.stats);
    return err;
}

cudaError_t launch_reduce(const ReduceArgs &args, int op, int dtype, int out_dtype, const LaunchShape &shape,
                          cudaStream_t stream, bool *supported)
{
    *supported = (dtype == kDtypeF32 || dtype == kDtypeBF16) && (out_dtype == kDtypeF32 || out_dtype == kDtypeBF16);
    if (!*supported) return cudaSuccess;
    return dtype == kDtypeF32 ? launch_reduce_f32(args, op, out_dtype, shape, stream) : launch_reduce_bf16(args, op, out_dtype, shape, stream);
}

}  // namespace wash
