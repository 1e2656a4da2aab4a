// One-time set-up per device (function attributes, checks of a compiled kernel), remembered only where it succeeded.
#pragma once

#include <atomic>

namespace sfb {

// ok(dev, setup) runs setup() until it has once returned true for that device and tells whether it has: after a set-up that
// failed every later call tries again, and a kernel behind it is never launched unchecked.  Two threads at once may both
// run it; it has to set the same values.
class PerDeviceOnce {
 public:
  template <typename F>
  bool ok(int dev, F&& setup) {
    const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;   // other ordinals: never remembered
    if (done_.load(std::memory_order_acquire) & bit) return true;
    if (!setup()) return false;
    done_.fetch_or(bit, std::memory_order_release);
    return true;
  }

 private:
  std::atomic<unsigned long long> done_{0};
};

}  // namespace sfb
