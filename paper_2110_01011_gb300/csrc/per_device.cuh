// Values that belong to a device (host code, no CUDA): what a kernel was
// configured with, how many of its CTAs are resident. A process may use several
// devices, so each is asked once per device and not once per process.
#pragma once

#include <atomic>
#include <mutex>

namespace rqlp {

template <typename T>
class PerDevice {
 public:
  // Device dev's value in *out; make(T*) finds it on the device's first use. Its
  // error code (0: found) is returned, and a device that failed is asked again.
  // (Devices beyond the table are asked every time.)
  template <typename F>
  int get(int dev, T* out, F make) {
    if (dev < 0 || dev >= kDevices) return make(out);
    Slot& s = slot_[dev];
    if (!s.found.load(std::memory_order_acquire)) {
      std::lock_guard<std::mutex> lk(mu_);
      if (!s.found.load(std::memory_order_relaxed)) {
        const int e = make(&s.value);
        if (e != 0) return e;
        s.found.store(true, std::memory_order_release);
      }
    }
    *out = s.value;
    return 0;
  }

 private:
  static constexpr int kDevices = 64;
  struct Slot {
    std::atomic<bool> found{false};
    T value{};
  };
  Slot slot_[kDevices];
  std::mutex mu_;
};

}  // namespace rqlp
