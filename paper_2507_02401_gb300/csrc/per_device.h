// A number that belongs to the current device (how many CTAs of a kernel it
// holds, say), worked out by the first call on that device and kept.
//
// Kernel attributes such as the dynamic shared-memory limit are set per device,
// and plans may live on several devices and be first used by several threads
// at once: so one entry per device, and an entry that several threads reach
// together is worked out by each of them (the work sets attributes and queries,
// it may be repeated) and stored atomically.  A failure (<= 0) is not kept.
#pragma once

#include <atomic>

namespace pat {

class PerDevice {
 public:
  static constexpr int kDevices = 64;

  // The kept value of `device`, or compute()'s.
  template <class F>
  int get(int device, F compute) {
    if (device < 0 || device >= kDevices) return compute();
    const int kept = value_[device].load(std::memory_order_acquire);
    if (kept > 0) return kept;
    const int v = compute();
    if (v > 0) value_[device].store(v, std::memory_order_release);
    return v;
  }

 private:
  std::atomic<int> value_[kDevices] = {};
};

}  // namespace pat
