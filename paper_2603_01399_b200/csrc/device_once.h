// What has to be done once, or asked once, on every device of a process (host code, no CUDA headers).
#pragma once

#include <stdint.h>

#include <atomic>

namespace quasar {

class DeviceOnce {
 public:
  // work() returns 0 when it has succeeded; it runs at the first call for `device`, and again while it has failed.  Threads that
  // come side by side may each run it: it has to be something that can be repeated.
  template <typename F>
  int run(int device, F&& work) {
    const bool kept = device >= 0 && device < 64;
    if (kept && ((done_.load(std::memory_order_acquire) >> device) & 1)) return 0;
    const int rc = work();
    if (rc == 0 && kept) done_.fetch_or((uint64_t)1 << device, std::memory_order_release);
    return rc;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

// Whole numbers that depend on nothing but the device: N questions.
template <int N>
class DeviceAnswers {
 public:
  // ask() returns a positive number, which is kept for `device`, or 0 where it could not be had: then the next call asks again.
  template <typename F>
  int get(int device, int question, F&& ask) {
    const bool kept = device >= 0 && device < 64 && question >= 0 && question < N;
    if (kept) {
      const int n = seen_[device][question].load(std::memory_order_relaxed);
      if (n > 0) return n;
    }
    const int n = ask();
    if (kept && n > 0) seen_[device][question].store(n, std::memory_order_relaxed);
    return n;
  }

 private:
  std::atomic<int> seen_[64][N] = {};
};

}  // namespace quasar
