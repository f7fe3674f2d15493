// Values that belong to a device: its number of SMs, a kernel's occupancy, a kernel's opt-in to more
// than 48 KiB of shared memory (cudaFuncSetAttribute acts on the current device only).  A process may
// use several devices and threads, so each value is made once per device, under a lock.
#pragma once

#include <map>
#include <mutex>

namespace bse {

template <typename T>
class PerDevice {
 public:
  // the value of device dev; make() runs with that device current
  template <typename Make>
  T get(int dev, Make make) {
    std::lock_guard<std::mutex> lock(mu_);
    auto it = v_.find(dev);
    if (it == v_.end()) it = v_.emplace(dev, make()).first;
    return it->second;
  }

 private:
  std::mutex mu_;
  std::map<int, T> v_;
};

}  // namespace bse
