// Values worked out once per GPU (internal; no CUDA in here).
#pragma once

#include <atomic>
#include <mutex>

namespace attn {

// Function attributes and occupancies belong to the device that is current when they are set or
// asked for, and a process may hold contexts on several. f() >= 0 is evaluated by the first caller
// on a device while others wait; one that throws leaves it to the next.
class PerDevice {
 public:
  static constexpr int kDevices = 64;
  template <class F>
  int get(int device, F f) {
    if (device < 0 || device >= kDevices) return f();
    int v = known_[device].load(std::memory_order_acquire);
    if (v == 0) {
      std::lock_guard<std::mutex> lock(mutex_);
      v = known_[device].load(std::memory_order_relaxed);
      if (v == 0) {
        v = f() + 1;
        known_[device].store(v, std::memory_order_release);
      }
    }
    return v - 1;
  }

 private:
  std::mutex mutex_;
  std::atomic<int> known_[kDevices] = {};  // value + 1, 0 while unknown
};

}  // namespace attn
