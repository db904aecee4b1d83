// per_device.cuh -- host state that belongs to a CUDA device.
#pragma once

#include <atomic>

namespace acpr {

// Devices on which something has been done: a kernel's attributes (shared
// memory, cluster size) hold on the device that was current when they were set.
// Threads may both find a device missing and both set it, to the same values.
class DeviceSet {
public:
    bool has(int dev) const { return dev >= 0 && dev < 64 && (bits_.load(std::memory_order_acquire) >> dev & 1); }
    void add(int dev) {
        if (dev >= 0 && dev < 64) bits_.fetch_or(1ULL << dev, std::memory_order_release);
    }

private:
    std::atomic<unsigned long long> bits_{0};
};

}  // namespace acpr
