// What is set up once per device: function attributes and the like hold for one
// device's context, so a flag per process would leave a second device without them.
#pragma once

#include <atomic>
#include <cstdint>

namespace bbl {

// One bit per device, set after the set-up has succeeded.  Threads may do the same
// set-up twice (it is idempotent); devices from 64 on do it on every call.
class OncePerDevice {
  public:
    bool need(int dev) const {
        return dev < 0 || dev >= 64 || !(bits_.load(std::memory_order_acquire) >> dev & 1u);
    }
    void done(int dev) {
        if (dev >= 0 && dev < 64) bits_.fetch_or(uint64_t(1) << dev, std::memory_order_release);
    }

  private:
    std::atomic<uint64_t> bits_{0};
};

}  // namespace bbl
