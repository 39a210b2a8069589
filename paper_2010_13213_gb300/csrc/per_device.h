// per_device.h -- work that is done once per device, such as setting a kernel's shared-memory limit: the attribute belongs
// to the device that is current when it is set.
#pragma once
#include <atomic>

namespace lgf {

class PerDevice {
  static constexpr int N = 64;
  std::atomic<bool> done[N] = {};

 public:
  // f() (true on success) for a device that it has not succeeded on yet; on return it has run on this device.  Two host
  // threads may both run it.
  template <class F>
  void run(int device, F f) {
    const bool known = device >= 0 && device < N;
    if (known && done[device].load(std::memory_order_acquire)) return;
    if (f() && known) done[device].store(true, std::memory_order_release);
  }
};

}  // namespace lgf
