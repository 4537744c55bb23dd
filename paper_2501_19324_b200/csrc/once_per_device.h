// Host-side bookkeeping without CUDA: what has to be done once for every device of the process.
#pragma once

#include <atomic>
#include <cstdint>

namespace rsd {

// A kernel's attributes belong to one device's context: set once per process, they were missing on the second device, and
// every launch there with more than 48 KB of shared memory failed.
class OncePerDevice {
 public:
  // Runs set() for `device` unless it has succeeded before (devices beyond 63: every time); its error, or 0.  Threads that
  // come at the same time may both run it.
  template <typename F> int run(int device, F set) {
    const bool noted = device >= 0 && device < 64;
    if (noted && ((done_.load(std::memory_order_acquire) >> device) & 1u)) return 0;
    const int e = set();
    if (e == 0 && noted) done_.fetch_or(uint64_t{1} << device, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace rsd
