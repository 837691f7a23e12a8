// A host-side setting that has to be made once per device: kernel attributes
// belong to the device that is current when they are set, so a cache of "this
// kernel is configured" is keyed by the device too.  Plain C++, no CUDA
// headers, so that a host test can check it without several GPUs.
#pragma once

#include <mutex>
#include <set>
#include <utility>

namespace kde {

class DeviceOnce {
 public:
  // set() unless it has succeeded (returned E(0)) for (device, key) before.
  template <typename E, typename F>
  E run(int device, const void* key, F&& set) {
    std::lock_guard<std::mutex> lk(mu_);
    if (done_.count({device, key})) return E(0);
    const E e = set();
    if (e == E(0)) done_.insert({device, key});
    return e;
  }

 private:
  std::mutex mu_;
  std::set<std::pair<int, const void*>> done_;
};

}  // namespace kde
