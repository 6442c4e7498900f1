// An action taken once per GPU of a process (host code without CUDA calls).
#pragma once

#include <atomic>

namespace pdep {

// Remembers the devices on which 'act' has succeeded (act returns 0 then): a
// kernel's shared-memory limit, for one, belongs to the device it was raised on.
// Devices past the 64th are not remembered, and a race of two threads acts twice.
class OncePerDevice {
  std::atomic<unsigned long long> done_{0};

 public:
  template <typename F>
  auto operator()(int device, F act) -> decltype(act()) {
    const bool kept = device >= 0 && device < 64;
    const unsigned long long bit = kept ? 1ull << device : 0ull;
    if (kept && (done_.load() & bit)) return decltype(act())(0);
    const auto r = act();
    if (r == decltype(act())(0) && kept) done_.fetch_or(bit);
    return r;
  }
};

}  // namespace pdep
