// A kernel that is launched with more than 48 KB of dynamic shared memory has to be opted in
// first, on every device it runs on: the attribute belongs to the kernel on the device that is
// current when it is set. One SmemOptIn per kernel (a static beside its launch) sets it the
// first time the kernel is launched on a device, which may be under stream capture (it is not a
// stream operation).
#pragma once
#include <cuda_runtime_api.h>
#include <stdint.h>

#include <atomic>

namespace stagkde {

class SmemOptIn {
    std::atomic<uint64_t> done_{0};  // bit i: set on device i

public:
    cudaError_t operator()(const void *kern, int bytes) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const uint64_t bit = dev < 64 ? 1ull << dev : 0;  // (beyond 64 devices: every time)
        if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
        return e;
    }
};

}  // namespace stagkde
