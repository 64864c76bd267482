// Something that has to be done once per GPU, such as raising a kernel's dynamic shared-memory limit, which holds for
// the device that is current.  Host code only (no CUDA).
#pragma once

#include <atomic>

namespace seedcg {

class DeviceOnce {
    static constexpr int kDevices = 64;
    std::atomic<bool> done_[kDevices] = {};

public:
    // set() unless it has returned for this device before; one that throws is tried again by the next call.  Two
    // threads may both call it, which is harmless for what is done here; devices past the table do it every time.
    template <typename Set>
    void run(int device, Set set) {
        const bool known = device >= 0 && device < kDevices;
        if (known && done_[device].load(std::memory_order_acquire)) return;
        set();
        if (known) done_[device].store(true, std::memory_order_release);
    }
};

}  // namespace seedcg
