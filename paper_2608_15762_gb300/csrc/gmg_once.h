// Set-up that holds for one device (a kernel's shared-memory limit): done once per
// device of the process, and again where it failed.
#pragma once

#include <mutex>

namespace gsim {

class OncePerDevice {
 public:
  // True if set() has succeeded for device `dev`, in this call or before.
  template <class F>
  bool done(int dev, F set) {
    if (dev < 0) return false;
    if (dev >= kMax) return set();
    std::lock_guard<std::mutex> lock(mu_);
    if (!ok_[dev]) ok_[dev] = set();
    return ok_[dev];
  }

 private:
  static constexpr int kMax = 64;
  std::mutex mu_;
  bool ok_[kMax] = {};
};

}  // namespace gsim
