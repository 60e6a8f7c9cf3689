// Set-up that a process does once on every device: the attributes of a kernel
// belong to the device that was current when they were set.  No CUDA here, so
// that it can be compiled and tested on a host.
#pragma once

#include <atomic>
#include <cstdint>

namespace spt {

// One object per kernel.  run(device, f) calls f until it has returned 0 (a
// success) on this device; devices from the 64th on call it every time.
class DeviceOnce {
  public:
    template <class F> int run(int device, F f)
    {
        const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;
        if (bit != 0 && (done_.load(std::memory_order_acquire) & bit) != 0) return 0;
        const int e = f();  // (two threads may both call it: it sets the same state)
        if (e == 0 && bit != 0) done_.fetch_or(bit, std::memory_order_release);
        return e;
    }

  private:
    std::atomic<uint64_t> done_{0};
};

}  // namespace spt
