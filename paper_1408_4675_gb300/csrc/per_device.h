// A positive number that is worked out once on each device, such as the CTAs per SM
// of a kernel, together with a kernel's attributes, which CUDA keeps per device.
// Any number of threads may ask at once: a number that is stored is final, and two
// threads that find none both work it out.
#pragma once

#include <atomic>

namespace kwgb {

class PerDevice {
    static constexpr int kDevices = 64;
    std::atomic<int> v_[kDevices] = {};               // 0: not worked out yet

public:
    // make() returns the number for the current device dev, or 0 if it failed (then the next call tries again)
    template <class Make>
    int get(int dev, Make&& make) {
        if (dev < 0 || dev >= kDevices) return make();
        int v = v_[dev].load(std::memory_order_acquire);
        if (v == 0) {
            v = make();
            v_[dev].store(v, std::memory_order_release);
        }
        return v;
    }
};

}  // namespace kwgb
