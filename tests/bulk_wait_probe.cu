// Test kernel: what the threads of a block are told about the block's bulk copies.
#include "wash_bulk_copy.cuh"

// The barrier expects nothing but one arrival, which comes first or (arrive == 0) never.
__global__ void probe(int arrive, uint32_t tries_first_warp, uint32_t tries, uint32_t *answer, long long *clocks)
{
    __shared__ __align__(8) unsigned long long s_barrier;
    __shared__ uint32_t s_gave_up;
    const uint32_t barrier = static_cast<uint32_t>(__cvta_generic_to_shared(&s_barrier));
    if (threadIdx.x == 0) {
        s_gave_up = 0;
        wash::bulk_barrier_init(barrier);
        if (arrive) wash::bulk_barrier_expect(barrier, 0);
    }
    __syncthreads();
    const long long start = clock64();
    answer[threadIdx.x] = wash::block_copies_done(barrier, threadIdx.x < 32 ? tries_first_warp : tries, &s_gave_up) ? 1u : 0u;
    clocks[threadIdx.x] = clock64() - start;
}

extern "C" int bulk_wait_probe(int arrive, uint32_t tries_first_warp, uint32_t tries, int threads, uint32_t *answer, long long *clocks)
{
    probe<<<1, threads>>>(arrive, tries_first_warp, tries, answer, clocks);
    const cudaError_t err = cudaGetLastError();
    return static_cast<int>(err != cudaSuccess ? err : cudaDeviceSynchronize());
}
