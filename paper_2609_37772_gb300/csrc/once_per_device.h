// Work done once for each device of a process, such as the opt-in of kernels to more than 48 KB of dynamic
// shared memory, which holds for the current device alone.
#pragma once
#include <mutex>

namespace uad {

class OncePerDevice {
 public:
  // f() for the first call of `dev`; its status, or 0 once it has returned 0. Calls that come meanwhile wait for it;
  // after a failure the next one tries again (and past kMax devices every one: f may be repeated). Nothing here throws
  // but what f does.
  template <class F>
  int run(int dev, F f) {
    std::lock_guard<std::mutex> lk(mu_);
    const bool known = dev >= 0 && dev < kMax;
    if (known && done_[dev]) return 0;
    const int rc = f();
    if (known) done_[dev] = rc == 0;
    return rc;
  }

 private:
  static constexpr int kMax = 64;
  std::mutex mu_;
  bool done_[kMax] = {};
};

}  // namespace uad
