// pfc_once.h -- something that has to be set once on each device.
#pragma once

#include <atomic>

namespace pfc {

// set() returns 0 where it succeeded; it runs on each device until it has, and
// may run twice where two threads meet (it must be idempotent).  Devices past
// 63 set it every time.
class OncePerDevice {
public:
    template <class Set>
    int operator()(int device, Set set)
    {
        const bool known = device >= 0 && device < kDevices;
        if (known && done_[device].load(std::memory_order_acquire)) return 0;
        const int e = set();
        if (known && e == 0) done_[device].store(true, std::memory_order_release);
        return e;
    }

private:
    static constexpr int kDevices = 64;
    std::atomic<bool> done_[kDevices] = {};
};

}  // namespace pfc
