// Work done once on each device of the process (host code only).
#pragma once

#include <stdint.h>

#include <atomic>

namespace pmnu {

// run(device, f) calls f until it has once returned true for that device.  A device is a bit of
// one word, so host threads need no lock (two that come first together may both call f, which has
// to be harmless); devices from 64 on call f every time.
class DeviceOnce {
  std::atomic<uint64_t> done{0};

 public:
  template <class F>
  void run(int device, F&& f) {
    const bool has_bit = device >= 0 && device < 64;
    const uint64_t bit = has_bit ? 1ull << device : 0;
    if (done.load(std::memory_order_acquire) & bit) return;
    if (f() && has_bit) done.fetch_or(bit, std::memory_order_release);
  }
};

}  // namespace pmnu
