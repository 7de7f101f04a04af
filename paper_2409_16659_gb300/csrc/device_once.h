// device_once.h -- work done once per device, by whichever thread comes
// first. Host code without CUDA calls of its own.
#pragma once

#include <atomic>
#include <mutex>

namespace mlsw {

// Runs f for device dev (0..63) unless a call for that device has succeeded
// (returned 0) before, and returns f's result, or 0. Whatever f stores is
// visible to every caller that gets 0.
class DeviceOnce {
 public:
  template <class F>
  auto operator()(int dev, F f) -> decltype(f()) {
    const unsigned long long bit = 1ull << dev;
    if (!(done_.load(std::memory_order_acquire) & bit)) {
      std::lock_guard<std::mutex> lock(mutex_);
      if (!(done_.load(std::memory_order_relaxed) & bit)) {
        const auto e = f();
        if (e != decltype(f()){}) return e;
        done_.fetch_or(bit, std::memory_order_release);
      }
    }
    return decltype(f()){};
  }

 private:
  std::atomic<unsigned long long> done_{0};
  std::mutex mutex_;
};

}  // namespace mlsw
