// How many blocks of a kernel fit an SM, looked up once per launch shape.
#pragma once
#include <cstdint>
#include <map>
#include <mutex>
#include <tuple>
#include <cuda_runtime.h>
#include "wash_internal.h"

namespace wash {

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
