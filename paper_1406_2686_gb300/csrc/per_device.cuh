// What a launch site sets up or asks once for a kernel: function attributes
// and occupancy belong to the device that is current, so once per device.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace vefd {

class PerDevice {
    static constexpr int kDevices = 64;  // devices beyond are set up at every call
    std::atomic<int> val_[kDevices] = {};

public:
    // *value of the current device, from make(value) at its first use there
    // (positive; not kept where make fails).  Threads that meet there both make it.
    template <class Make>
    cudaError_t get(int* value, Make make) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const bool kept = dev >= 0 && dev < kDevices;
        *value = kept ? val_[dev].load(std::memory_order_acquire) : 0;
        if (*value > 0) return cudaSuccess;
        e = make(value);
        if (e == cudaSuccess && kept) val_[dev].store(*value, std::memory_order_release);
        return e;
    }
};

// Allows `bytes` of dynamic shared memory for a kernel on the current device.
template <class K>
cudaError_t allow_smem(PerDevice& site, K kernel, int bytes) {
    int done = 0;
    return site.get(&done, [&](int* v) {
        *v = 1;
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    });
}

}  // namespace vefd
