// A host-side number per device, found on its first use there: how many CTAs
// of a kernel a device holds, once the kernel has been allowed its dynamic
// shared memory there (an attribute that the runtime keeps per device).
#pragma once

#include <atomic>

namespace s2d {

class PerDevice {
 public:
  static constexpr int MAX_DEVICES = 64;

  // Device `dev`'s number: find() on the first use, which gives the same on
  // every call (threads that come together may each call it).  Numbers below 1
  // are failures, and not kept.
  template <typename F>
  int get(int dev, F find) {
    if (dev < 0 || dev >= MAX_DEVICES) return find();
    int n = n_[dev].load(std::memory_order_acquire);
    if (n < 1) {
      n = find();
      if (n >= 1) n_[dev].store(n, std::memory_order_release);
    }
    return n;
  }

 private:
  std::atomic<int> n_[MAX_DEVICES] = {};
};

}  // namespace s2d
