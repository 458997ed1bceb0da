// Host-side values that belong to a device, not to the process: a kernel's shared-memory limit (set once
// per device), how many clusters fit.
#pragma once
#include <atomic>

namespace chem {

// get(dev, f): the positive value that f() gave for device dev the first time; f runs again as long as it
// gives 0 or less (a failure is not kept).  Safe from several threads (f may run in more than one of them
// at first, with the same result); devices past the table run f every time.
class PerDevice {
 public:
  template <typename F>
  int get(int dev, F f) {
    const bool kept = dev >= 0 && dev < kDevices;
    if (kept) {
      const int v = v_[dev].load(std::memory_order_acquire);
      if (v > 0) return v;
    }
    const int v = f();
    if (kept && v > 0) v_[dev].store(v, std::memory_order_release);
    return v;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<int> v_[kDevices] = {};
};

}  // namespace chem
