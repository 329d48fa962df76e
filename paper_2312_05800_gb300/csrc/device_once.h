// device_once.h -- host values that belong to a device: a kernel's dynamic shared memory limit is set for
// the current device only, and the SM count is that device's. Keyed by the device index, for any
// number of threads; plain C++.
#pragma once

#include <atomic>
#include <stdint.h>

namespace chemgb {

constexpr int kMaxDevices = 64;         // indices beyond are set and looked up on every call

// Runs set() (0 = success) once per device; again after a failure.
class DeviceOnce {
    std::atomic<uint64_t> done_{0};

public:
    template <class F>
    int run(int dev, F &&set) {
        const bool keyed = dev >= 0 && dev < kMaxDevices;
        if (keyed && (done_.load(std::memory_order_acquire) >> dev & 1u)) return 0;
        const int rc = set();
        if (rc == 0 && keyed) done_.fetch_or(uint64_t(1) << dev, std::memory_order_release);
        return rc;
    }
};

// A positive integer of each device, looked up by get() once per device.
class DeviceInt {
    std::atomic<int> v_[kMaxDevices]{};

public:
    template <class F>
    int value(int dev, F &&get) {
        if (dev < 0 || dev >= kMaxDevices) return get();
        int v = v_[dev].load(std::memory_order_relaxed);
        if (v <= 0) {
            v = get();
            v_[dev].store(v, std::memory_order_relaxed);
        }
        return v;
    }
};

}  // namespace chemgb
