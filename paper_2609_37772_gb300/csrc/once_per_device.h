// Work done once for each device of a process, such as the opt-in of kernels to more than 48 KB of dynamic
// shared memory, which holds for the current device alone.
#pragma once
#include <mutex>
#include <set>

namespace uad {

class OncePerDevice {
 public:
  // f() for the first call of `dev`; its status, or 0 once it has returned 0. Calls that come meanwhile wait for it;
  // after a failure the next one tries again.
  template <class F>
  int run(int dev, F f) {
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

}  // namespace uad
