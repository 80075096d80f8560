// A value made once for each CUDA device, by whichever thread asks for it
// first: a kernel's attributes and its occupancy belong to a device, and
// contexts on several devices and threads share the library.
#pragma once

#include <atomic>
#include <mutex>

namespace wdc {

template <class T>
class PerDevice {
public:
    static constexpr int kDevices = 64;        // above, the value is made on every call

    // make(T&) fills the value and returns whether to keep it; one that is not
    // kept (a query failed) is made again by the next call.
    template <class Make>
    T get(int device, Make make) {
        T v{};
        if (device < 0 || device >= kDevices) {
            make(v);
            return v;
        }
        if (ready_[device].load(std::memory_order_acquire)) return value_[device];
        std::lock_guard<std::mutex> lock(mu_);
        if (ready_[device].load(std::memory_order_relaxed)) return value_[device];
        if (make(v)) {
            value_[device] = v;
            ready_[device].store(true, std::memory_order_release);
        }
        return v;
    }

private:
    std::mutex mu_;
    std::atomic<bool> ready_[kDevices]{};
    T value_[kDevices]{};
};

}  // namespace wdc
