// A number set up once per device: a grid that fits, a kernel's attribute in
// place.  Function attributes and occupancy belong to a device, so what one
// device was given says nothing about another.
#pragma once

#include <atomic>

namespace crc {

class PerDevice {
public:
    // The value of device dev, from make() when it has none yet: > 0 a value, < 0
    // a refusal (both are kept), 0 a failure, tried again by the next call.
    // Threads that meet may each call make(); devices past the table always do.
    template <class F>
    int get(int dev, F make) {
        if (dev < 0 || dev >= kDevices) return make();
        int v = value_[dev].load(std::memory_order_acquire);
        if (v == 0) {
            v = make();
            value_[dev].store(v, std::memory_order_release);
        }
        return v;
    }
    void set(int dev, int v) {
        if (dev >= 0 && dev < kDevices) value_[dev].store(v, std::memory_order_release);
    }

private:
    static constexpr int kDevices = 64;
    std::atomic<int> value_[kDevices] = {};
};

}  // namespace crc
