// Private: a set-up that is made once on every device.
#pragma once

#include <atomic>

namespace dgm {

// once(dev, setup) runs setup() unless it has succeeded on device dev before,
// and returns its status (0: success).  Host threads may call it together: two
// that both find it undone both run setup(), which has to be repeatable.
// Devices beyond the array set up on every call.
class OncePerDevice {
    static constexpr int kDevices = 64;
    std::atomic<bool> done_[kDevices] = {};

public:
    template <class F>
    int operator()(int dev, F &&setup) {
        const bool known = dev >= 0 && dev < kDevices;
        if (known && done_[dev].load(std::memory_order_acquire)) return 0;
        const int st = setup();
        if (known && st == 0) done_[dev].store(true, std::memory_order_release);
        return st;
    }
};

}  // namespace dgm
