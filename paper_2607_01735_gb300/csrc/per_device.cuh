// A value that belongs to a CUDA device and not to the process: a kernel's raised shared-memory
// limit, an SM count, an occupancy.  Computed once for each device, by the first call with that
// device current, safely from several threads.
#pragma once

#include <cuda_runtime.h>

#include <mutex>

namespace rbgs {

template <typename T>
class PerDevice {
public:
    template <typename F>
    T get(F compute) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) {
            cudaGetLastError();
            return compute();
        }
        if (dev < 0 || dev >= kDevices) return compute();
        std::call_once(once_[dev], [&] { value_[dev] = compute(); });
        return value_[dev];
    }

private:
    static constexpr int kDevices = 64;  // past these every call computes
    std::once_flag once_[kDevices];
    T value_[kDevices] = {};
};

// Raises a kernel's dynamic shared-memory limit on the current device, once for each; a failure is
// reported on every call.  `set`: one object per kernel, with static storage.
template <typename Kernel>
cudaError_t raise_smem(PerDevice<cudaError_t> &set, Kernel *kernel, size_t bytes) {
    return set.get([&] {
        const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) cudaGetLastError();
        return e;
    });
}

}  // namespace rbgs
