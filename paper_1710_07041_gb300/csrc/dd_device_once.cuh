// Work done once per device, such as raising a kernel's shared-memory limit,
// which the CUDA runtime keeps for the current device only. A try that fails is
// not remembered: the next call tries again. Any thread may call it.
#pragma once
#include <mutex>
#include <set>

namespace dd {

class DeviceOnce {
 public:
  // f() for device `dev` unless one of its calls there has returned 0; its result
  template <typename F> int run(int dev, F f) {
    std::lock_guard<std::mutex> lk(mu_);
    if (done_.count(dev)) return 0;
    const int rc = f();
    if (rc == 0) done_.insert(dev);
    return rc;
  }

 private:
  std::mutex mu_;
  std::set<int> done_;
};

}  // namespace dd
