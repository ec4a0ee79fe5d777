// Work done once per device of the process (plain C++, no CUDA headers).
#pragma once

#include <atomic>
#include <mutex>

namespace edpc {

// run(dev, f) calls f until it has once returned zero (success) for device
// ordinal dev. Kernel attributes and memory pools belong to one device's
// context, so a flag per process would leave every device but the first
// without them. Safe to call from any thread; ordinals beyond kDevices, which
// no flag is kept for, call f every time.
class OncePerDevice {
 public:
  static constexpr int kDevices = 64;
  template <class F>
  auto run(int dev, F&& f) -> decltype(f()) {
    using R = decltype(f());
    const bool kept = dev >= 0 && dev < kDevices;
    if (kept && done_[dev].load(std::memory_order_acquire)) return R{};
    std::lock_guard<std::mutex> lock(mu_);
    if (kept && done_[dev].load(std::memory_order_relaxed)) return R{};
    const R r = f();
    if (kept && r == R{}) done_[dev].store(true, std::memory_order_release);
    return r;
  }

 private:
  std::atomic<bool> done_[kDevices] = {};
  std::mutex mu_;
};

}  // namespace edpc
