// One int per device, found on first use, for launches from any host thread.
#pragma once
#include <atomic>

namespace vg {

class DeviceInt {
 public:
  static constexpr int kDevices = 64;
  // The device's value; find() gives it (0: none) unless an earlier call has.  Threads that meet
  // here on first use may both call find(), and store the same.
  template <typename Find>
  int get(int dev, Find find) {
    if (dev < 0 || dev >= kDevices) return 0;
    int v = value_[dev].load(std::memory_order_acquire);
    if (v == 0) {
      v = find();
      if (v <= 0) v = -1;
      value_[dev].store(v, std::memory_order_release);
    }
    return v > 0 ? v : 0;
  }

 private:
  std::atomic<int> value_[kDevices] = {};
};

}  // namespace vg
