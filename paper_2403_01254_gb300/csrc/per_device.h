// A positive number worked out once per device and kept for the process: what a kernel's
// launch needs that belongs to the device (an opt-in to more shared memory, the CTAs that fit).
// Host code without CUDA headers.
#pragma once

#include <atomic>

namespace rk {

class PerDevice {
public:
    // The number of device `dev`: make()'s, called again until it is positive.  Threads that
    // meet in the first call each make it (make() gives each the same).
    template <typename Make>
    int get(int dev, Make make) {
        const bool kept = dev >= 0 && dev < MAX;
        int v = kept ? v_[dev].load(std::memory_order_acquire) : 0;
        if (v > 0) return v;
        v = make();
        if (kept && v > 0) v_[dev].store(v, std::memory_order_release);
        return v;
    }

private:
    static constexpr int MAX = 64;     // devices beyond are asked each time
    std::atomic<int> v_[MAX] = {};
};

}  // namespace rk
