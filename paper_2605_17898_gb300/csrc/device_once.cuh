// What has been done once per device (a kernel's attributes belong to the device that was current when they were set), safe
// with several threads. Plain C++, shared with its host check.
#pragma once

#include <atomic>
#include <cstdint>

namespace lgp {

class DeviceOnce {
  public:
    // Whether add(device) has been called. Never for devices beyond 63: there the work is repeated.
    bool has(int device) const { return device >= 0 && device < 64 && (done_.load(std::memory_order_acquire) >> device & 1u); }
    // After the work has succeeded.
    void add(int device) {
        if (device >= 0 && device < 64) done_.fetch_or(uint64_t(1) << device, std::memory_order_release);
    }

  private:
    std::atomic<uint64_t> done_{0};
};

}  // namespace lgp
