// Host side: settings that a device needs once, before the first launch of a kernel there.  Plain C++.
#pragma once
#include <atomic>
#include <utility>

namespace flop {

constexpr int kMaxDevices = 64;

// `set` runs before the call returns, unless it has already run to success for the device.  The mark is made after it, not before: a
// thread that found the mark of a setting still under way would launch its kernel without it.  Two threads may run `set` at the
// same time (function attributes may be set twice); a failed one is tried again by the next call.
class OncePerDevice {
 public:
  template <typename F>
  int operator()(int dev, F&& set) {           // dev < 0: unknown device, set every time
    const bool known = dev >= 0 && dev < kMaxDevices;
    if (known && done_[dev].load(std::memory_order_acquire)) return 0;
    const int rc = std::forward<F>(set)();
    if (known && rc == 0) done_[dev].store(true, std::memory_order_release);
    return rc;
  }

 private:
  std::atomic<bool> done_[kMaxDevices] = {};
};

}  // namespace flop
