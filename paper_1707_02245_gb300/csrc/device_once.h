// Something to be done once per device of the process: attributes of a kernel, for instance, are
// kept per device, so setting them for the device current at a first call leaves the others without.
#pragma once

#include <atomic>
#include <mutex>

namespace pat {

class DeviceOnce {
public:
    // set() (0 on success) unless it has succeeded for device dev before; a failure is returned and
    // tried again by the next call.  Devices past the table are set every time.
    template <class F>
    int run(int dev, F set) {
        if (dev < 0 || dev >= kDevices) return set();
        if (done_[dev].load(std::memory_order_acquire)) return 0;
        std::lock_guard<std::mutex> lock(mtx_);
        if (done_[dev].load(std::memory_order_relaxed)) return 0;
        const int e = set();
        if (e == 0) done_[dev].store(true, std::memory_order_release);
        return e;
    }

private:
    static constexpr int kDevices = 64;
    std::mutex mtx_;
    std::atomic<bool> done_[kDevices] = {};
};

}  // namespace pat
