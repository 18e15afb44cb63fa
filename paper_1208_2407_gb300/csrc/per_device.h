// A value of the current CUDA device (function attributes, occupancy, counts),
// made at the first use on that device.
#pragma once

#include <cuda_runtime.h>
#include <mutex>

namespace ts {

template <typename T>
class PerDevice {
    static constexpr int kDevices = 64;
    std::once_flag made_[kDevices];
    T value_[kDevices];

public:
    template <typename F>
    const T &get(F make)
    {
        int dev = -1;
        cudaGetDevice(&dev);
        if (dev < 0 || dev >= kDevices) {   // no such device: made each time
            thread_local T value;
            return value = make();
        }
        std::call_once(made_[dev], [&] { value_[dev] = make(); });
        return value_[dev];
    }
};

}  // namespace ts
