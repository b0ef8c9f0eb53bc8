// kite_once.h -- host values computed once per device.
#pragma once

#include <atomic>

namespace kite {

// A value >= 0 kept per device: a kernel's launch attributes (its dynamic shared-memory limit,
// set on the way) and what follows from them belong to one device, so a value kept per process
// leaves the kernels of a second device's context at the default limit.  A negative value is
// returned but not kept.  Threads may compute the same value side by side.
class PerDevice {
 public:
  template <typename F>
  int get(int device, F compute) {
    if (device < 0 || device >= kDevices) return compute();
    int v = kept_[device].load(std::memory_order_acquire) - 1;
    if (v < 0) {
      v = compute();
      if (v >= 0) kept_[device].store(v + 1, std::memory_order_release);
    }
    return v;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<int> kept_[kDevices] = {};  // value + 1, 0: none yet
};

}  // namespace kite
