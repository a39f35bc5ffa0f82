// Launching a kernel in the chain of a stream, and how many blocks of one fit an SM (looked up once per
// launch shape).
#pragma once
#include <cstdint>
#include <map>
#include <mutex>
#include <tuple>
#include <cuda_runtime.h>
#include "wash_internal.h"

namespace wash {

// Kernels of this library are launched with the programmatic-serialization attribute: a launch need not
// wait until the kernel before it in the stream has drained, its blocks may start as that one's
// last blocks run.  In return every kernel calls await_previous() before it touches anything that an
// earlier kernel may write or read -- which waits until the kernels before it are complete and their
// writes visible.  A kernel of another library launched in the ordinary way, or a copy, is ordered as always; one that is
// itself launched as a programmatic dependent has to wait, too, before it reads a stack (include/wash.h says so).
//
// let_next_start() allows the next kernel's blocks to be placed.  Two rules for where it is called:
//   after await_previous(): called before, a chain of short launches piles up, kernel after kernel resident and waiting, and the
//     blocks of the one whose turn comes sit several to an SM (EMA of 16 bf16 models, 2^17 coordinates, back to back
//     7.2 us without programmatic launches, 13.9 released first, 6.4 released after the wait; 20 models, [P][N] 8.3, 20.6, 10.2).
//     Kernels whose work before the wait is what the overlap is for say so themselves.
//   by the last blocks only: a release takes the launch unit about a nanosecond, a block after the other, which is more than
//     a block of the one-trip streaming kernel takes of the memory: five models, 2^24 coordinates, p = 1e-4 53 us without, 70
//     with a release in every block, 51 from the last kReleasing.  A block that ends without it counts as released, so the
//     next kernel starts no later; no more blocks than these are resident at a time.
constexpr unsigned kReleasing = 148 * 32;
__device__ __forceinline__ void await_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start()
{
    if (gridDim.x - blockIdx.x <= kReleasing) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... Params, class... Args>
cudaError_t launch_chained(void (*kernel)(Params...), unsigned grid, unsigned threads, size_t smem, cudaStream_t stream, const Args &...args)
{
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t config = {};
    config.gridDim = dim3(grid);
    config.blockDim = dim3(threads);
    config.dynamicSmemBytes = smem;
    config.stream = stream;
    config.attrs = &attr;
    config.numAttrs = 1;
    cudaError_t err = cudaLaunchKernelEx(&config, kernel, static_cast<Params>(args)...);
    if (err == cudaSuccess) count_launch();
    return err;
}

struct KernelFit {
    int occupancy;   // resident blocks per SM at (threads, smem)
};

inline cudaError_t kernel_fit(const void *kernel, int threads, size_t smem, KernelFit *fit)
{
    static std::mutex mu;
    static std::map<std::tuple<const void *, int, size_t, int>, KernelFit> cache;
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    const auto key = std::make_tuple(kernel, threads, smem, dev);
    {
        std::lock_guard<std::mutex> lock(mu);
        auto it = cache.find(key);
        if (it != cache.end()) { *fit = it->second; return cudaSuccess; }
    }
    if (smem > 32 * 1024) {   // static shared memory counts against the default 48 KiB too
        // raise the kernel's limit to the device's opt-in maximum (never lower it: other
        // launch shapes of the same kernel may already rely on a larger value)
        int optin = 0;
        err = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
        if (err != cudaSuccess) return err;
        optin -= 1024;   // room for the kernels' few bytes of static shared memory
        if (optin < 0 || smem > static_cast<size_t>(optin)) return cudaErrorInvalidConfiguration;
        err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
        if (err != cudaSuccess) return err;
    }
    int occ = 0;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem);
    if (err != cudaSuccess) return err;
    KernelFit f{occ};
    {
        std::lock_guard<std::mutex> lock(mu);
        cache[key] = f;
    }
    *fit = f;
    return cudaSuccess;
}

}  // namespace wash
