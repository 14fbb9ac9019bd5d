// A value made once for each device and kept: what the runtime keeps for a kernel (its shared
// memory opt-in, how many of its blocks are resident) belongs to the device that was current when
// it was set or asked for, not to the process.
#pragma once
#include <atomic>

namespace dtg {

struct PerDevice {
  static constexpr int kDevices = 64;
  std::atomic<long long> value[kDevices] = {};  // what make() returned plus one; 0: not made yet

  // The value of device `dev`, from make() (>= 0) the first time. Two threads may both make it; a
  // device beyond the table gets a new one each time.
  template <class F>
  long long get(int dev, F make) {
    if (dev < 0 || dev >= kDevices) return make();
    long long v = value[dev].load(std::memory_order_acquire);
    if (v == 0) {
      v = (long long)make() + 1;
      value[dev].store(v, std::memory_order_release);
    }
    return v - 1;
  }
};

}  // namespace dtg
