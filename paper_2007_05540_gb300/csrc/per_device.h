// A kernel's shared-memory limit, raised once per device: the attribute belongs to the device that is current when
// it is set, not to the process.
#pragma once

#include <atomic>
#include <cstdint>

namespace heff {

// Marks for devices 0 .. 63; a device beyond them is never marked.
class PerDevice {
    std::atomic<uint64_t> mask_{0};

public:
    bool marked(int device) const {
        return device >= 0 && device < 64 && ((mask_.load(std::memory_order_acquire) >> device) & 1u);
    }
    void mark(int device) {
        if (device >= 0 && device < 64) mask_.fetch_or(uint64_t(1) << device, std::memory_order_release);
    }
};

// raise(): sets the limit on the current device and returns its status (0: done).  `done` belongs to the kernel.
template <class Raise>
int once_per_device(PerDevice& done, int device, Raise raise) {
    if (done.marked(device)) return 0;
    const int status = raise();
    if (status == 0) done.mark(device);
    return status;
}

}  // namespace heff
