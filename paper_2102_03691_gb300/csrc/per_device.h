// Set-up that CUDA wants once on every device.  A kernel's attributes (its shared-memory opt-in, its
// largest cluster) belong to the device that is current when they are set, so a process that uses
// several devices has to set them on each.  Host code only.
#pragma once
#include <atomic>
#include <cstdint>

namespace mhc {

// once(device, set): runs `set` unless it has succeeded on that device (numbers from 64 on are set
// at every call).  A failure is returned and not kept, so the next call tries again.  Threads that
// meet on a device's first call may both run `set`, which has to allow it (setting an attribute does).
class PerDevice {
    std::atomic<uint64_t> done_{0};

public:
    template <typename Set>
    auto operator()(int device, Set set) -> decltype(set()) {
        using Error = decltype(set());
        const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;
        if (done_.load(std::memory_order_acquire) & bit) return Error{};
        const Error e = set();
        if (e == Error{}) done_.fetch_or(bit, std::memory_order_release);
        return e;
    }
};

}  // namespace mhc
