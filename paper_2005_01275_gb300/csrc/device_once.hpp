// What has to be done or asked once on every device of the process (kernel attributes belong to a device's context).
#pragma once
#include <atomic>

namespace nlmg {

class DeviceOnce {
 public:
  // Runs f (returns 0 on success) on device dev unless it has succeeded there before; any thread, any number of devices (on
  // those beyond the table f runs every time). Threads that arrive together may both run it.
  template <class F>
  auto run(int dev, F&& f) -> decltype(f()) {
    const bool known = dev >= 0 && dev < kDevices;
    if (known && done_[dev].load(std::memory_order_acquire)) return decltype(f())(0);
    const auto e = f();
    if (known && e == decltype(f())(0)) done_[dev].store(true, std::memory_order_release);
    return e;
  }
  static constexpr int kDevices = 64;

 private:
  std::atomic<bool> done_[kDevices] = {};
};

}  // namespace nlmg
