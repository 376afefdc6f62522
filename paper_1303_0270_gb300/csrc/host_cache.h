// host_cache.h -- facts of a device that the launchers keep between calls (an
// occupancy, a kernel attribute that has been set), because asking again costs
// more than a launch.  Calls come from several threads and for several devices.
#pragma once

#include <atomic>

namespace ccm {

// One positive number per device.  Threads that ask at the same time each ask
// the device and store the same answer; a failed question is not kept.
class DeviceCache {
 public:
  // The kept number of device `dev`; else ask()'s, kept when positive; else `otherwise`.
  template <class Ask>
  int get(int dev, int otherwise, Ask ask) {
    const bool keeps = dev >= 0 && dev < kDevices;
    if (keeps) {
      const int kept = value_[dev].load(std::memory_order_acquire);
      if (kept > 0) return kept;
    }
    const int got = ask();
    if (got <= 0) return otherwise;
    if (keeps) value_[dev].store(got, std::memory_order_release);
    return got;
  }

 private:
  static constexpr int kDevices = 32;
  std::atomic<int> value_[kDevices] = {};
};

}  // namespace ccm
