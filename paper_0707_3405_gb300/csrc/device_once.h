// What is done once on each device (plain C++: the caller names the device).
#pragma once

#include <atomic>
#include <cstdint>

namespace lg {

// A function's attributes hold for the device that was current when they were set, so the flag of a
// kernel's shared-memory limit is kept by device.  Several threads may find it clear and set the same
// limit; devices from 64 on set it at every call.
class DeviceOnce {
    std::atomic<uint64_t> done_{0};

public:
    bool done(int dev) const { return dev >= 0 && dev < 64 && (done_.load() >> dev & 1) != 0; }
    void mark(int dev) {
        if (dev >= 0 && dev < 64) done_.fetch_or(uint64_t(1) << dev);
    }
};

}  // namespace lg
