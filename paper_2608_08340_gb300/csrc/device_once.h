// Work to be done once per device of a process, such as raising a kernel's
// shared memory limit (the attribute belongs to the current device's context).
#pragma once

#include <atomic>
#include <cstdint>

namespace oprag {

// One bit per device for the first 64; further ones do the work every time.
class DeviceOnce {
 public:
  // Runs work() (0 = success) unless it has succeeded on `device`.  Two threads
  // may run it at the same time on a device's first call.
  template <typename Work>
  auto run(int device, Work&& work) -> decltype(work()) {
    const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;
    if (done_.load(std::memory_order_acquire) & bit) return decltype(work())(0);
    const auto rc = work();
    if (rc == decltype(work())(0)) done_.fetch_or(bit, std::memory_order_release);
    return rc;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace oprag
