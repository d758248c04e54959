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

// alloc(n) for a group of n items, and where memory for so many is not to be had (`short_of`) for half as many, down to
// one; n is the size it succeeded with, or that of another failure.
template <typename R, typename F>
R fit_group(int& n, R short_of, F&& alloc) {
  for (;;) {
    const R r = alloc(n);
    if (r != short_of || n <= 1) return r;
    n = (n + 1) / 2;
  }
}
