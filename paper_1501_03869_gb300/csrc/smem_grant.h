// smem_grant.h -- the largest dynamic shared memory a kernel was granted, per
// device, in plain C++ so that a host test can check it (internal).
#pragma once

#include <cstddef>
#include <mutex>

namespace patbp {

// The attribute belongs to a device and may only grow: a launch that needs less
// than another thread's must not take back what that one relies on.
class SmemGrant {
 public:
  // Calls set(bytes) for the current device `dev` where it has less so far.
  template <class Set>
  auto ensure(int dev, size_t bytes, Set set) -> decltype(set(bytes)) {
    using E = decltype(set(bytes));
    const std::lock_guard<std::mutex> lk(mu_);
    if (dev < 0 || dev >= kDevices) return set(bytes);
    if (bytes <= granted_[dev]) return E{};
    const E e = set(bytes);
    if (e == E{}) granted_[dev] = bytes;
    return e;
  }

 private:
  static constexpr int kDevices = 64;
  std::mutex mu_;
  size_t granted_[kDevices] = {};
};

}  // namespace patbp
