// State that belongs to a device and is made at its first use there (kernel
// attributes, device properties): one value per device, safe with several host
// threads.  Host code only, without CUDA calls of its own.
#pragma once

#include <map>
#include <mutex>

namespace cbddc {

template <typename T>
class PerDevice {
  std::mutex mu_;
  std::map<int, T> made_;

 public:
  // The value of device dev, from make() if it has none yet.  Callers of the same
  // device wait for one that is being made; after an exception the next call
  // tries again.
  template <typename F>
  T get(int dev, F&& make) {
    std::lock_guard<std::mutex> lock(mu_);
    auto it = made_.find(dev);
    if (it != made_.end()) return it->second;
    T v = make();
    made_.emplace(dev, v);
    return v;
  }
};

}  // namespace cbddc
