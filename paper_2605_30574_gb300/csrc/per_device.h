// Launch state that belongs to a device: kernel attributes that are set, and
// counts that are queried, at the first launch on each.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>

namespace splice {

template <class T>
class PerDevice {
public:
    // The current device's state.  make(device, &state) sets it up at the
    // device's first use (threads that come at once may each do so) and returns
    // a cudaError_t; a failure is returned, with the runtime's record of it
    // cleared, and not kept.
    template <class Make>
    cudaError_t get(T* out, Make&& make) {
        int dev = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess && dev < kDevices && made_[dev].load(std::memory_order_acquire) == kMade) {
            *out = state_[dev];
            return cudaSuccess;
        }
        if (e == cudaSuccess) e = make(dev, out);
        if (e != cudaSuccess) {
            cudaGetLastError();
            return e;
        }
        int none = 0;
        if (dev < kDevices && made_[dev].compare_exchange_strong(none, kMaking)) {
            state_[dev] = *out;
            made_[dev].store(kMade, std::memory_order_release);
        }
        return cudaSuccess;
    }

private:
    static constexpr int kDevices = 64;          // (those past it are set up at every call)
    static constexpr int kMaking = 1, kMade = 2;
    T state_[kDevices] = {};
    std::atomic<int> made_[kDevices] = {};
};

}  // namespace splice
