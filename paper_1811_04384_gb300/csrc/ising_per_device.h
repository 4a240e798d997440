// A setup that belongs to a device: kernel attributes and occupancy are those of
// the current device's copy of a kernel, so a process that uses several devices
// makes each its own.
#pragma once
#include <cuda_runtime.h>

#include <mutex>

namespace ising {

template <typename T>
class PerDevice {
public:
    // make()'s result on the current device, made at the first call there.  An
    // error that make() leaves behind is cleared: its result says what failed.
    template <typename Make>
    T get(Make make)
    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) {
            cudaGetLastError();
            return T();
        }
        std::lock_guard<std::mutex> lock(mutex_);
        if (!made_[dev]) {
            value_[dev] = make();
            cudaGetLastError();
            made_[dev] = true;
        }
        return value_[dev];
    }

private:
    static constexpr int kDevices = 64;
    std::mutex mutex_;
    bool made_[kDevices] = {};
    T value_[kDevices] = {};
};

}  // namespace ising
