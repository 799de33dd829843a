// A number that belongs to a device (the dynamic shared memory its kernels may take), kept per device.
#pragma once

#include <atomic>

namespace pdg {

// get(dev, make): make() the first time it is asked for on device dev, that value from then on.  Threads that ask
// at once may each call make; it has to give all of them the same positive value.
class PerDevice {
    static constexpr int kDevices = 64;   // (a device beyond these is asked each time)
    std::atomic<int> value_[kDevices] = {};

public:
    template <class F>
    int get(int dev, F&& make) {
        if (dev < 0 || dev >= kDevices) return make();
        int v = value_[dev].load(std::memory_order_acquire);
        if (v == 0) {
            v = make();
            value_[dev].store(v, std::memory_order_release);
        }
        return v;
    }
};

}  // namespace pdg
