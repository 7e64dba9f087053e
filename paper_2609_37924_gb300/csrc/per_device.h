// What a launcher sets up once per device and keeps: a kernel's opt-in shared
// memory is an attribute of the kernel on one device, and the SM count is the
// device's own, so a process that changes its current device needs both again.
#pragma once
#include <atomic>
#include <mutex>

namespace tadm {

class PerDevice {
 public:
  static constexpr int kMax = 64;
  // The value (> 0) of device `dev`.  `setup` makes it on the first call for
  // that device, one thread at a time; a result <= 0 is handed to the caller
  // and not kept, so the next call tries again.  A device past kMax is set up
  // on every call.
  template <class F>
  int get(int dev, F&& setup) {
    if (dev < 0 || dev >= kMax) return setup();
    int v = val_[dev].load(std::memory_order_acquire);
    if (v > 0) return v;
    std::lock_guard<std::mutex> lock(mu_);
    v = val_[dev].load(std::memory_order_relaxed);
    if (v > 0) return v;
    v = setup();
    if (v > 0) val_[dev].store(v, std::memory_order_release);
    return v;
  }

 private:
  std::mutex mu_;
  std::atomic<int> val_[kMax] = {};
};

}  // namespace tadm
