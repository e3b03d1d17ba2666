// What a process sets up once on each device, whichever thread comes first.
#pragma once

#include <atomic>
#include <cstdint>

namespace fwi {

// A function attribute holds on the device that was current when it was set, so a
// process that uses two GPUs has to set it on both.  Every instantiation of a kernel
// keeps one of these (static storage); two threads may both find a device not done and
// set the same value twice.  Devices beyond the 64th are set on every launch.
class DeviceOnce {
 public:
  bool done(int dev) const {
    return dev >= 0 && dev < 64 && (mask_.load(std::memory_order_acquire) >> dev & 1u) != 0;
  }
  void mark(int dev) {
    if (dev >= 0 && dev < 64) mask_.fetch_or(uint64_t{1} << dev, std::memory_order_release);
  }

 private:
  std::atomic<uint64_t> mask_{0};
};

}  // namespace fwi
