// Dynamic shared memory beyond 48 KB, which a kernel has to be allowed per device.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace tdg {

// One per kernel: sets the attribute once on each device that is current at a launch,
// and again after a failure.
struct SmemOptIn {
    std::atomic<uint64_t> done{0};       // bit per device ordinal below 64
    template <typename Kern>
    cudaError_t allow(Kern kern, int bytes) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;
        if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_release);
        return e;
    }
};

}  // namespace tdg
