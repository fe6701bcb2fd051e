// Opt-in of a kernel to more than 48 KB of dynamic shared memory.
//
// The limit belongs to a (kernel, device) pair and outlives the call that sets it, so
// it is never set to one launch's own size: two threads whose launches differ could
// then leave the smaller of two limits behind the larger one's record.  Every caller
// sets the same value, all that the device lets the kernel have (its static shared
// memory taken off), and a device is recorded only after its limit is in place.  The
// limit itself costs nothing: occupancy and the L1 split follow a launch's own size.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace omm {

// One object per kernel (a function-local static of its launcher).
class SmemOptIn {
   public:
    template <class K>
    cudaError_t operator()(K *kernel) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const uint64_t bit = dev < 64 ? 1ull << dev : 0ull;   // past 64 devices: set it every time
        if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
        int most = 0;
        cudaFuncAttributes at{};
        if ((e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess ||
            (e = cudaFuncGetAttributes(&at, (const void *)kernel)) != cudaSuccess ||
            (e = cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      most - (int)at.sharedSizeBytes)) != cudaSuccess)
            return e;
        done_.fetch_or(bit, std::memory_order_release);
        return cudaSuccess;
    }

   private:
    std::atomic<uint64_t> done_{0};   // bit d: device d
};

}  // namespace omm
