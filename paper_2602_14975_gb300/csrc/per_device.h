// Figures that depend on the device alone (SM count, resident blocks), found
// once for each device a process uses. Host code without CUDA calls.
#pragma once
#include <atomic>

namespace dmts {

class PerDevice {
public:
    // find() for device `dev`, a positive number; safe from several threads
    // (they store the same value).
    template <class Find>
    int get(int dev, Find find) {
        if (dev < 0 || dev >= kDevices) return find();
        int v = value_[dev].load(std::memory_order_relaxed);
        if (v == 0) value_[dev].store(v = find(), std::memory_order_relaxed);
        return v;
    }

private:
    static constexpr int kDevices = 64;
    std::atomic<int> value_[kDevices] = {};
};

}  // namespace dmts
