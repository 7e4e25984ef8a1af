// Set-up that every device needs once (host code only; safe from several threads).
#pragma once
#include <atomic>
#include <cstdint>

namespace shweno {

// Which devices have been set up.  Beyond 64 none is remembered: the set-up then runs every time.
class DeviceOnce {
 public:
  bool needed(int dev) const { return dev < 0 || dev >= 64 || !(done_.load(std::memory_order_acquire) >> dev & 1); }
  void done(int dev) {
    if (dev >= 0 && dev < 64) done_.fetch_or(uint64_t(1) << dev, std::memory_order_release);
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace shweno
