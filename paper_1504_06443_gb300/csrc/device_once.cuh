// Settings and facts that belong to a device context, made or asked once per device, from any host thread.
// Plain C++.
#pragma once
#include <atomic>
#include <cstdint>
#include <mutex>

namespace gep {

constexpr int MAX_DEVICES = 64;

// run(dev, f) calls f once for a device.  A thread that finds it under way waits until it is done, so nobody goes
// on before it is; an f that does not return 0 is tried again by the next call.
class DeviceOnce {
  std::atomic<uint64_t> done_{0};
  std::mutex m_;

 public:
  template <class F>
  int run(int dev, F&& f) {
    if (dev < 0 || dev >= MAX_DEVICES) return f();
    const uint64_t bit = (uint64_t)1 << dev;
    if (done_.load(std::memory_order_acquire) & bit) return 0;
    std::lock_guard<std::mutex> lock(m_);
    if (done_.load(std::memory_order_relaxed) & bit) return 0;
    const int rc = f();
    if (rc == 0) done_.fetch_or(bit, std::memory_order_release);
    return rc;
  }
};

// A number per device: get(dev, &v, f) sets v to what f(&v) found the first time.
class DeviceValue {
  DeviceOnce once_;
  int value_[MAX_DEVICES] = {};

 public:
  template <class F>
  int get(int dev, int* v, F&& f) {
    if (dev < 0 || dev >= MAX_DEVICES) return f(v);
    const int rc = once_.run(dev, [&]() { return f(&value_[dev]); });
    *v = value_[dev];
    return rc;
  }
};

}  // namespace gep
