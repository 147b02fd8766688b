// once_per_device.h -- set-up that belongs to a function or a symbol and a device.
#pragma once
#include <cuda_runtime.h>
#include <atomic>

namespace spgb {

// Run `set` on the current device unless it ran there before (in this process): for
// what belongs to a function or a symbol and a device, as the opt-in to more shared
// memory.  done: a static of the caller with a bit per device; threads that come at
// the same time may both run `set`.
template <typename F> cudaError_t once_per_device(std::atomic<unsigned long long> &done, F &&set)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ULL << dev : 0;
    if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
    if ((e = set()) == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
    return e;
}
inline cudaError_t opt_in_smem(const void *kernel, size_t bytes, std::atomic<unsigned long long> &done)
{
    return once_per_device(done, [&] {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    });
}

}  // namespace spgb
