// Host-side bookkeeping of steps that belong to a device.
#pragma once

#include <atomic>
#include <cstdint>

namespace deer {

// A step to be done once per device, such as setting an attribute of a kernel: attributes belong
// to a device's context, so a process (or thread) that goes on to another device does the step
// there too. A failed step is tried again by the next call; devices past the 64th do it on every
// call. Safe from several threads, which at worst repeat the step.
class DeviceOnce {
 public:
  // the status of `step` (0 = success), or 0 where it has succeeded on `device` before
  template <class Step>
  auto ensure(int device, Step step) -> decltype(step()) {
    using Status = decltype(step());
    const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;
    if (done_.load(std::memory_order_acquire) & bit) return Status(0);
    const Status st = step();
    if (st == Status(0)) done_.fetch_or(bit, std::memory_order_release);
    return st;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace deer
