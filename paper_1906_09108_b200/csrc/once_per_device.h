// Settings that belong to a device (a kernel's shared-memory limit) and are made the first time that one needs them: once
// per device, from any number of host threads.
#pragma once
#include <stdint.h>

#include <atomic>

namespace fdg {

// Runs `work` (returning 0 on success) unless it has succeeded for device `dev` before.  When this returns 0, `work` has been
// completed for that device.  Threads that meet here at the same time may each run it: it has to bear that.  A failure is
// not remembered.  Devices past the 64th are not remembered either.
class OncePerDevice {
 public:
  template <typename Work> auto run(int dev, Work work) -> decltype(work()) {
    const uint64_t bit = dev >= 0 && dev < 64 ? (uint64_t)1 << dev : 0;
    if (done_.load(std::memory_order_acquire) & bit) return decltype(work())(0);
    const auto e = work();
    if (e == decltype(work())(0)) done_.fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace fdg
