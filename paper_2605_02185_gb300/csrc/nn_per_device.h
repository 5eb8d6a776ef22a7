// nn_per_device.h -- a number found once per device: kernel attributes belong to the
// device they were set on, so "set once" means once on each.
#pragma once

#include <atomic>

namespace gbnn_tc {

struct PerDevice {
  static constexpr int kDevices = 64;  // beyond them it is found anew on every call
  std::atomic<int> value[kDevices] = {};

  // find() on the first call for `device` (two threads may both make it) and again while
  // it gives 0 or less, which is not kept.
  template <class Find>
  int get(int device, Find find) {
    if (device < 0 || device >= kDevices) return find();
    int v = value[device].load(std::memory_order_acquire);
    if (v <= 0) {
      v = find();
      if (v > 0) value[device].store(v, std::memory_order_release);
    }
    return v;
  }
};

}  // namespace gbnn_tc
