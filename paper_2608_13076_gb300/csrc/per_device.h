// per_device.h -- work that a process does once per device, whichever thread comes first.
#pragma once
#include <atomic>

namespace spade {

constexpr int kMaxDevices = 64;

// Runs `set` (0: success) the first time that device `dev` is asked for, and returns
// its error; a failure is not remembered.  Threads that come first together may
// run it twice.
class OncePerDevice {
 public:
  template <class F>
  auto operator()(int dev, F set) -> decltype(set()) {
    const bool kept = dev >= 0 && dev < kMaxDevices;
    if (kept && done_[dev].load(std::memory_order_acquire)) return decltype(set()){};
    const auto e = set();
    if (kept && e == decltype(set()){}) done_[dev].store(true, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<bool> done_[kMaxDevices] = {};
};

}  // namespace spade
