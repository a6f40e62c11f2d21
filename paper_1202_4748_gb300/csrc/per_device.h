// A small value computed once per device: function attributes (shared-memory
// limits, carve-outs) belong to the device that was current when they were set, so
// a second device of the same process needs them again.  Safe with several threads
// (they may compute the same value at once; it is the same value).  Plain C++.
#pragma once

#include <atomic>

namespace lbf {

class PerDevice {
    static constexpr int kDevices = 64;
    std::atomic<signed char> value_[kDevices] = {};

public:
    // f() for this device, kept when it is not 0 (0: failed, asked again next time)
    template <class F>
    int get(int device, F&& f) {
        const bool kept = device >= 0 && device < kDevices;
        if (kept) {
            const int v = value_[device].load(std::memory_order_acquire);
            if (v) return v;
        }
        const int v = f();
        if (kept && v) value_[device].store(static_cast<signed char>(v), std::memory_order_release);
        return v;
    }
};

}  // namespace lbf
