// tk_device_once.h -- settings that CUDA keeps per device and function.
//
// A kernel's opt-in to more than 48 KB of dynamic shared memory holds on the device
// that is current when it is made; a process may hold solvers on several.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace tk {

// set() once for each device that is current at a call (again where it failed);
// devices from 64 on each time.  Constant-initialised: a function-local static.
class DeviceOnce {
    std::atomic<unsigned long long> done_{0};

public:
    template <class Set>
    cudaError_t operator()(Set set)
    {
        int dev = 0;
        const cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const unsigned long long bit = dev < 64 ? 1ull << dev : 0;
        if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
        const cudaError_t s = set();
        if (s == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
        return s;
    }
};

// The opt-in of a kernel, whose once it is.
inline cudaError_t allow_smem(DeviceOnce &once, const void *kern, size_t bytes)
{
    return once([&] {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    });
}

}  // namespace tk
