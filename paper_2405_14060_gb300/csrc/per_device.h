// Launch preparation that belongs to a device and not to the process: the
// shared memory a kernel may use beyond 48 KB, and values read from the device.
#pragma once
#include <atomic>
#include <cstdint>

namespace tn {

// once(dev, f) runs f on the first call for each device.  Two threads that meet
// on a device's first call may both run it, so f must bear repetition; no call
// returns before f has run once for its device.
class PerDevice {
  public:
    template <typename F>
    void once(int dev, F &&f) {
        const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0;   // beyond: every call
        if (bit && (seen_.load(std::memory_order_acquire) & bit)) return;
        f();
        seen_.fetch_or(bit, std::memory_order_release);
    }

  private:
    std::atomic<uint64_t> seen_{0};
};

}  // namespace tn
