// Something that has to be done once on every device (host code).
#pragma once
#include <atomic>
#include <cstdint>

namespace sky {

// Calls f for a device until it has returned 0 there once, and returns what it
// returned, else 0.  Threads may call it together (f may then run more than once).
class OncePerDevice {
 public:
  template <class F>
  auto operator()(int device, F&& f) -> decltype(f()) {
    // ordinals past the mask: every time
    const uint64_t bit = device >= 0 && device < 64 ? uint64_t{1} << device : 0;
    if (done_.load(std::memory_order_acquire) & bit) return decltype(f()){};
    const auto e = f();
    if (e == decltype(f()){}) done_.fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace sky
