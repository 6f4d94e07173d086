// One-time set-up per device: kernel attributes hold for the device that is
// current when they are set, so that each device that a process uses needs them
// once.  Safe from several threads (two that come first may both do it).
#pragma once
#include <cuda_runtime.h>

#include <atomic>

namespace tdse {

class DeviceOnce {
public:
    // f(), returning a cudaError_t, unless it has succeeded on the current device.
    template <class F> cudaError_t operator()(F f) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0;
        if (done_.load(std::memory_order_acquire) & bit) return cudaSuccess;
        e = f();
        if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_release);
        return e;
    }

private:
    std::atomic<unsigned long long> done_{0};
};

}  // namespace tdse
