// Set-up that CUDA keeps per device (a kernel's attributes): done once on each device
// that uses it, from whichever thread comes first, and again after a failure.
#pragma once
#include <atomic>
#include <mutex>

namespace ifd {

class DeviceOnce {
  static constexpr int MOST = 64;  // devices remembered; beyond, the set-up is repeated
  std::mutex lock_;
  std::atomic<bool> done_[MOST] = {};

 public:
  // Whether `device` is set up; set_up() returns whether it succeeded.
  template <class F>
  bool operator()(int device, F &&set_up) {
    if (device < 0 || device >= MOST) return set_up();
    if (done_[device].load(std::memory_order_acquire)) return true;
    const std::lock_guard<std::mutex> hold(lock_);
    if (!done_[device].load(std::memory_order_relaxed) && set_up())
      done_[device].store(true, std::memory_order_release);
    return done_[device].load(std::memory_order_relaxed);
  }
};

}  // namespace ifd
