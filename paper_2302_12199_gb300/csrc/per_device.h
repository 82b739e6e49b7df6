// A launcher's value for each device: kernel attributes (the opt-in to more
// shared memory, the carveout) and the blocks that fit belong to a device, so
// they are set and found on each device that a process launches on, once.
#pragma once
#include <atomic>
#include <climits>
#include <mutex>

namespace mstgpu {

class PerDevice {
 public:
  PerDevice() {
    for (auto &v : value_) v.store(UNSET, std::memory_order_relaxed);
  }
  // The value of device `dev` (the current one): find()'s the first time, kept
  // from then on.  Host threads that come at the same time wait for it.  An
  // ordinal past the table is asked for every time.
  template <class Find>
  int get(int dev, Find &&find) {
    if (dev < 0 || dev >= DEVICES) return find();
    int v = value_[dev].load(std::memory_order_acquire);
    if (v != UNSET) return v;
    std::lock_guard<std::mutex> hold(lock_);
    v = value_[dev].load(std::memory_order_relaxed);
    if (v == UNSET) {
      v = find();
      value_[dev].store(v, std::memory_order_release);
    }
    return v;
  }

 private:
  static constexpr int DEVICES = 64, UNSET = INT_MIN;
  std::atomic<int> value_[DEVICES];
  std::mutex lock_;
};

}  // namespace mstgpu
