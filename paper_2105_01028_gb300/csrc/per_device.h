// Set-up that belongs to a device (a kernel's shared-memory limit, the SM count), made on
// first use there.  Contexts of one process may live on several devices and be driven from
// several host threads.
#pragma once

#include <mutex>

namespace trinity {

constexpr int kMaxDevices = 64;

class PerDevice {
 public:
  // What set_up() returned on the first use of device ``dev``; 0 says that it failed (the
  // next call tries again) or that there is no such device.
  template <class F>
  int get(int dev, F set_up) {
    if (dev < 0 || dev >= kMaxDevices) return 0;
    std::lock_guard<std::mutex> lk(mu_);
    if (value_[dev] == 0) value_[dev] = set_up();
    return value_[dev];
  }

 private:
  std::mutex mu_;
  int value_[kMaxDevices] = {};
};

}  // namespace trinity
