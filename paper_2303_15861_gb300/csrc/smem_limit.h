// More than 48 KB of dynamic shared memory has to be allowed for each kernel on each device.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace adr {

// One per kernel (function-local static): allows it `bytes` on the current device the first time a launch asks there.
// A failure is reported to that launch alone.
class SmemLimit {
    std::atomic<unsigned long long> devices_{0};             // those that have it, ordinals below 64

public:
    cudaError_t allow(const void* kernel, int bytes) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
        if (devices_.load(std::memory_order_acquire) & bit) return cudaSuccess;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess) devices_.fetch_or(bit, std::memory_order_release);
        return e;
    }
};

}  // namespace adr
