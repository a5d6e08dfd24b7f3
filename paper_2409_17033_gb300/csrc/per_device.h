// Host-side values that belong to one GPU (a kernel's resident block count, set up
// together with its shared-memory limit, which is an attribute of the kernel on one
// device): filled at a device's first use, by one thread, and kept for that device.
#pragma once
#include <atomic>
#include <mutex>

namespace sp2 {

constexpr int kMaxDevices = 64;

class PerDevice {
 public:
  // *value of device `dev`, from fill(int* value) at its first use. fill returns 0 and a
  // value above 0, or an error, which is returned (and nothing kept); a device out of
  // range returns `bad`.
  template <typename E, typename F>
  E get(int dev, E bad, int* value, F fill) {
    if (dev < 0 || dev >= kMaxDevices) return bad;
    *value = v_[dev].load(std::memory_order_acquire);
    if (*value > 0) return E(0);
    std::lock_guard<std::mutex> lock(mu_);
    *value = v_[dev].load(std::memory_order_relaxed);
    if (*value > 0) return E(0);
    const E e = fill(value);
    if (e != E(0)) return e;
    v_[dev].store(*value, std::memory_order_release);
    return E(0);
  }

 private:
  std::atomic<int> v_[kMaxDevices] = {};
  std::mutex mu_;
};

}  // namespace sp2
