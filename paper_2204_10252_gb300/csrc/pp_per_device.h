// Results that belong to a device: kernel attributes, occupancies.
#pragma once
#include <atomic>

namespace pp {

// A number worked out by the first call on each device and kept for the life of the
// process.  `work` returns it (0 or more), or a negative number when it failed: then
// nothing is kept and the next call tries again.  Calls from several threads may work
// it out at the same time, so `work` has to bear being repeated.
class PerDevice {
  public:
    template <class F> int get(int device, F&& work) {
        if (device < 0 || device >= kDevices) return work();
        const int kept = kept_[device].load(std::memory_order_acquire);
        if (kept > 0) return kept - 1;
        const int v = work();
        if (v >= 0) kept_[device].store(v + 1, std::memory_order_release);
        return v;
    }

  private:
    static constexpr int kDevices = 64;
    std::atomic<int> kept_[kDevices] = {};
};

}  // namespace pp
