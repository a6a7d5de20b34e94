// Facts about a device that the host asks the runtime once per process and reads at every launch: multiprocessors, resident
// blocks of a kernel, clusters that fit.
#pragma once
#include <atomic>
#include <mutex>

namespace he {

constexpr int kMaxDevices = 64;

// One non-zero value per device and item, worked out by the first caller and read by every later one, from any thread.
// `make(int*)` runs under the lock and returns 0 or an error code, which is handed on; the next caller then tries again.
template <int ITEMS>
class DeviceTable {
 public:
  template <typename F>
  int get(int dev, int item, int* out, F make) {
    std::atomic<int>& at = value_[dev][item];
    int v = at.load(std::memory_order_acquire);
    if (v == 0) {
      std::lock_guard<std::mutex> lock(mu_);
      v = at.load(std::memory_order_relaxed);
      if (v == 0) {
        if (int rc = make(&v)) return rc;
        at.store(v, std::memory_order_release);
      }
    }
    *out = v;
    return 0;
  }

 private:
  std::atomic<int> value_[kMaxDevices][ITEMS] = {};
  std::mutex mu_;
};

}  // namespace he
