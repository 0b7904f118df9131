// A value of the host side that is found once per device (a launch attribute
// set, an occupancy), kept for the process.
#ifndef DQT_PER_DEVICE_H_
#define DQT_PER_DEVICE_H_

#include <atomic>

namespace dqt {

// compute(value) finds the value (not 0) and returns whether it could; the
// devices beyond the table find theirs on each call.  Threads that meet a
// device for the first time together may each compute it, and each sees only
// whole values.
class PerDevice {
 public:
  template <typename F>
  bool get(int dev, int& value, F&& compute) {
    const bool kept = dev >= 0 && dev < kDevices;
    if (kept) {
      value = v_[dev].load(std::memory_order_acquire);
      if (value != 0) return true;
    }
    int fresh = 0;
    if (!compute(fresh) || fresh == 0) return false;
    if (kept) v_[dev].store(fresh, std::memory_order_release);
    value = fresh;
    return true;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<int> v_[kDevices] = {};
};

}  // namespace dqt

#endif  // DQT_PER_DEVICE_H_
