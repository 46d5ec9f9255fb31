// A kernel's opt-in to more dynamic shared memory than 48 KB, once per device:
// the attribute belongs to the device that is current when it is set, so one
// flag for the process leaves a second device's launches to fail.  Plain C++ (the call that
// sets the attribute is the caller's), so that it can be checked without a GPU.
#pragma once

#include <stddef.h>

#include <atomic>
#include <mutex>

namespace lsp {

class SmemOptIn {
 public:
  // Make sure that `bytes` are granted on `device`: 0, or what set() returned.  Only success
  // is remembered.  Any thread may call it.
  template <typename F>
  int ensure(int device, size_t bytes, F set) {
    if (device < 0 || device >= kDevices) return set();
    std::atomic<size_t>& granted = granted_[device];
    if (granted.load(std::memory_order_acquire) >= bytes) return 0;
    std::lock_guard<std::mutex> lock(mu_);
    if (granted.load(std::memory_order_relaxed) >= bytes) return 0;
    const int e = set();
    if (e == 0) granted.store(bytes, std::memory_order_release);
    return e;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<size_t> granted_[kDevices] = {};
  std::mutex mu_;
};

}  // namespace lsp
