// device_once.h -- what has to be done once per device of the process, such as
// a kernel's opt-in to more shared memory (an attribute of the device current
// at the call).  Plain C++.
#pragma once
#include <atomic>

class DeviceOnce {
 public:
  // act() (0: done) on the first call for this device, and again while it
  // fails; several threads may act at once, which an attribute's setting
  // allows.  Devices beyond kDevices act on every call.
  template <class F>
  int operator()(int dev, F act) {
    const bool known = dev >= 0 && dev < kDevices;
    if (known && done_[dev].load(std::memory_order_acquire)) return 0;
    const int e = act();
    if (e == 0 && known) done_[dev].store(true, std::memory_order_release);
    return e;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<bool> done_[kDevices] = {};
};
