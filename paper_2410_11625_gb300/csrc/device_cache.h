// device_cache.h -- values of a device that launches need and that do not change while the process
// runs (how many CTAs of a kernel are resident, that a kernel's attributes are set, the number of
// SMs): formed once per device, by one thread.  Host code without CUDA.
#pragma once

#include <atomic>
#include <mutex>

// get(dev, fill, out): the value of device dev, from fill(value) on its first call, which returns 0
// (success) or an error code that get passes on; a failed fill is tried again by the next call.
// One instance serves every thread.  Looking a filled value up takes one load and a copy.
template <class T>
class PerDevice {
    static constexpr int kDevices = 64;
    std::mutex mu_;
    std::atomic<bool> ready_[kDevices] = {};
    T value_[kDevices] = {};

public:
    template <class F>
    auto get(int dev, F fill, T &out) -> decltype(fill(out))
    {
        using E = decltype(fill(out));
        if (dev < 0 || dev >= kDevices) return fill(out);
        if (!ready_[dev].load(std::memory_order_acquire)) {
            std::lock_guard<std::mutex> lock(mu_);
            if (!ready_[dev].load(std::memory_order_relaxed)) {
                const E e = fill(value_[dev]);
                if (e != E(0)) return e;
                ready_[dev].store(true, std::memory_order_release);
            }
        }
        out = value_[dev];
        return E(0);
    }
};
