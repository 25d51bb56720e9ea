// Once per device, for settings that the CUDA runtime keeps per function and device (the limit
// of dynamic shared memory).  Plain C++.
#pragma once
#include <atomic>

namespace gbmg {

// The devices (0 .. 63) that a setting has been made on.
using DeviceSet = std::atomic<unsigned long long>;

// set() on the device's first call, and again after a failure (a value other than zero) or on
// devices beyond the set; safe with several threads, which may each set the same value.
template <class Set>
auto once_per_device(DeviceSet& done, int device, Set set) -> decltype(set()) {
  using R = decltype(set());
  const unsigned long long bit = device >= 0 && device < 64 ? 1ull << device : 0;
  if (done.load(std::memory_order_acquire) & bit) return R();
  const R r = set();
  if (r == R()) done.fetch_or(bit, std::memory_order_release);
  return r;
}

}  // namespace gbmg
