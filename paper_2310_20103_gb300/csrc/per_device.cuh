// What is set or asked for once per device.  A kernel's attributes belong to
// the device that was current when they were set: a process whose handles are
// on two devices needs them on both, and its threads may come together.
#pragma once

#include <atomic>

namespace lgw {

constexpr int MAX_DEVICES = 64;   // above this, every call does the work again

struct DeviceOnce {
  std::atomic<unsigned long long> done{0};
  // f() before the first return for this device; f may run again where threads
  // meet, and must not mind.
  template <class F>
  void operator()(int dev, F f) {
    const bool known = dev >= 0 && dev < MAX_DEVICES;
    const unsigned long long bit = known ? 1ull << dev : 0;
    if (done.load(std::memory_order_acquire) & bit) return;
    f();
    done.fetch_or(bit, std::memory_order_release);
  }
};

struct DeviceValue {
  std::atomic<int> v[MAX_DEVICES] = {};
  // f(), which is positive, kept for the device
  template <class F>
  int operator()(int dev, F f) {
    const bool known = dev >= 0 && dev < MAX_DEVICES;
    if (known) {
      const int x = v[dev].load(std::memory_order_relaxed);
      if (x > 0) return x;
    }
    const int x = f();
    if (known) v[dev].store(x, std::memory_order_relaxed);
    return x;
  }
};

}  // namespace lgw
