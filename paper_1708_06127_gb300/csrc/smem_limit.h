// Which kernels already have a raised dynamic shared-memory limit, and where: the limit is an
// attribute of the kernel on one device, so it is raised once per kernel and device.
#pragma once
#include <stddef.h>

#include <map>
#include <mutex>
#include <utility>

namespace vc {

class SmemLimits {
 public:
  // Calls raise() unless an earlier one that returned gave `kernel` at least `bytes` on `device`.
  template <typename F>
  void require(const void* kernel, int device, size_t bytes, F raise) {
    std::lock_guard<std::mutex> lock(mu_);
    auto it = limit_.find({kernel, device});
    if (it != limit_.end() && it->second >= bytes) return;
    raise();
    limit_[{kernel, device}] = bytes;
  }

 private:
  std::mutex mu_;
  std::map<std::pair<const void*, int>, size_t> limit_;
};

}  // namespace vc
