// once_per_device.h -- host-side set-up that a process needs once for each of its devices (the opt-in of a kernel to
// more than 48 KB of dynamic shared memory belongs to the function on the current device).  Plain C++.
#pragma once

#include <stdint.h>

#include <atomic>

namespace nh {

class OncePerDevice {
public:
    // set() (a status, zero for success) unless it has succeeded for this device before.  Threads that come at the same
    // time may both run it, so it has to be harmless twice; from device 64 on it always runs.
    template <typename F>
    auto operator()(int device, F&& set) -> decltype(set())
    {
        using Status = decltype(set());
        const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;
        if (done_.load(std::memory_order_acquire) & bit) return Status{};
        const Status s = set();
        if (s == Status{}) done_.fetch_or(bit, std::memory_order_release);
        return s;
    }

private:
    std::atomic<uint64_t> done_{0};
};

}  // namespace nh
