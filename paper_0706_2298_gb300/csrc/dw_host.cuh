// Host helpers that need no CUDA declarations.
#pragma once

#include <atomic>
#include <cstdint>

// Something to be done once on each device (a kernel's shared-memory limit): f(), which returns 0 for success, runs
// until it has succeeded for `device`; a failure is not kept.
class DeviceOnce {
  std::atomic<uint64_t> done_[4] = {};

 public:
  template <typename F>
  auto operator()(int device, F&& f) -> decltype(f()) {
    using R = decltype(f());
    const bool known = device >= 0 && device < 256;
    const uint64_t bit = (uint64_t)1 << (device & 63);
    if (known && (done_[device >> 6].load(std::memory_order_acquire) & bit)) return R{};
    const R r = f();
    if (known && r == R{}) done_[device >> 6].fetch_or(bit, std::memory_order_release);
    return r;
  }
};
