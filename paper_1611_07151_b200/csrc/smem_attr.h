// Permission for more than 48 KB of dynamic shared memory, per kernel and device.
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace sqn {

// One (static) object per kernel.  The attribute belongs to the kernel on one device: set once in a process, launches on a
// second device were refused.  Calls may come from several threads; setting it twice does no harm.
class SmemAttr {
public:
    cudaError_t allow(const void* kernel, size_t bytes)
    {
        int dev = 0;
        cudaError_t rc = cudaGetDevice(&dev);
        if (rc != cudaSuccess) return rc;
        const uint64_t bit = dev >= 0 && dev < 64 ? (uint64_t)1 << dev : 0;       // (beyond 64 devices: at every launch)
        if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
        rc = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (rc == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
        return rc;
    }

private:
    std::atomic<uint64_t> done_{0};
};

}  // namespace sqn
