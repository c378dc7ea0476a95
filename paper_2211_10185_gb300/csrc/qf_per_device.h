// Work that a process does once on each of its devices, such as raising a kernel's shared-memory
// limit or finding out whether a cluster fits: both are properties of a function on a device.
#pragma once
#include <atomic>
#include <mutex>

namespace qf {

class PerDevice {
 public:
  // Result of setup() on device `dev`: called the first time for each device, by one thread.
  template <typename F>
  bool ready(int dev, F&& setup) {
    if (dev < 0 || dev >= kMax) return setup();
    signed char s = state_[dev].load(std::memory_order_acquire);
    if (s == 0) {
      std::lock_guard<std::mutex> lock(mu_);
      s = state_[dev].load(std::memory_order_relaxed);
      if (s == 0) {
        s = setup() ? 1 : -1;
        state_[dev].store(s, std::memory_order_release);
      }
    }
    return s > 0;
  }

 private:
  static constexpr int kMax = 64;
  std::mutex mu_;
  std::atomic<signed char> state_[kMax] = {};  // 0 not known, 1 ready, -1 not to be had
};

}  // namespace qf
