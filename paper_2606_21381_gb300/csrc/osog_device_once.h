// A step of host set-up that the CUDA runtime keeps per device (a kernel's
// shared-memory opt-in, say), run once on each.
//
// Header of plain C++, so that the host can check it.
#pragma once

#include <stdint.h>

#include <atomic>

namespace osog {

// One per step (static storage).  Threads that meet on a device's first call may
// each run the step; a failure is not remembered.
class DeviceOnce {
  public:
    // set_up() (an error code, 0 on success) unless it has succeeded on `device`.
    template <typename F>
    auto operator()(int device, F set_up) -> decltype(set_up()) {
        using Error = decltype(set_up());
        if (device < 0 || device >= 64) return set_up();
        const uint64_t bit = (uint64_t)1 << device;
        if (done_.load(std::memory_order_acquire) & bit) return Error(0);
        const Error e = set_up();
        if (e == Error(0)) done_.fetch_or(bit, std::memory_order_release);
        return e;
    }

  private:
    std::atomic<uint64_t> done_{0};
};

}  // namespace osog
