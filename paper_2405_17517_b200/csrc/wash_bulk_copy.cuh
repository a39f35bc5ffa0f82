// Bulk copies of a block's contiguous bytes into its shared memory, and the wait for them.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace wash {

// By one thread, before its first copy: the barrier, and the bytes that its copies will bring.
__device__ __forceinline__ void bulk_barrier_init(uint32_t barrier)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(barrier) : "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void bulk_barrier_expect(uint32_t barrier, uint32_t bytes)
{
    asm volatile("{\n\t.reg .b64 s;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 s, [%0], %1;\n\t}" ::"r"(barrier), "r"(bytes) : "memory");
}

// A copy by one thread (16-byte aligned, a multiple of 16 bytes), reported to the barrier.
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t barrier)
{
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes), "r"(barrier) : "memory");
}

// Waits for the barrier's first phase, but not for ever: `tries` trials.  A trial that sees nothing arrive returns after 7850 clocks, so
// kBulkTries are a second (1.05 s at 1.965 GHz); copies take microseconds.
constexpr uint32_t kBulkTries = 1u << 18;
__device__ __forceinline__ bool bulk_copies_done(uint32_t barrier, uint32_t tries)
{
    for (uint32_t i = 0; i < tries; ++i) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(barrier) : "memory");
        if (done) return true;
    }
    return false;
}

// The same for the block, called by all of its threads, and a barrier for them: every thread gets one answer, so that a wait that one of
// them gives up lets none move a value (a part of an exchange loses values and doubles others).  *gave_up (shared) is zero before.  The word read behind the barrier costs N =
// 32 fp32, 2^25, p = 0.1 708.5 -> 713 us; a vote in the barrier 714-715, a count that only threads that gave up look at 716.
__device__ __forceinline__ bool block_copies_done(uint32_t barrier, uint32_t tries, volatile uint32_t *gave_up)
{
    if (!bulk_copies_done(barrier, tries)) *gave_up = 1u;
    __syncthreads();
    return *gave_up == 0u;
}

}  // namespace wash
