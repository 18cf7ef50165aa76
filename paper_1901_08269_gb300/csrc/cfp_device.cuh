// State that belongs to a device rather than to the process (host code only).
#pragma once

#include <atomic>

namespace cfp {

// Work to be done once on every device, such as setting a kernel's function
// attributes: run(dev, f) calls f unless it has returned 0 for dev before.
// Several threads may call it at once; f must be harmless when run twice
// (two threads may both find it not done) and runs every time on a device
// beyond the table.
class OncePerDevice {
  public:
    template <class F>
    auto run(int dev, F f) -> decltype(f()) {
        const bool kept = dev >= 0 && dev < kDevices;
        if (kept && done_[dev].load(std::memory_order_acquire)) return decltype(f())(0);
        const auto st = f();
        if (kept && st == decltype(f())(0)) done_[dev].store(true, std::memory_order_release);
        return st;
    }

  private:
    static constexpr int kDevices = 64;
    std::atomic<bool> done_[kDevices] = {};
};

}  // namespace cfp
