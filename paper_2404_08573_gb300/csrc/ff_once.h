// Settings that hold per device, made once on each device that is used.
#pragma once

#include <atomic>

namespace ff {

// The status of set() on the current device (get(&index) names it), run
// unless it has succeeded there before; done: one bit per device index, zero
// at first.  A failure is not kept: the next call tries again.  set() may run
// twice when threads race, so it has to be repeatable.
template <typename Status, typename Get, typename Set>
Status once_per_device(std::atomic<unsigned long long>& done, Get get, Set set) {
  int dev = -1;
  Status s = get(&dev);
  if (s != Status{}) return s;
  const unsigned long long bit = dev >= 0 && dev < 64 ? 1ull << dev : 0;  // devices past 63: every time
  if (done.load(std::memory_order_acquire) & bit) return Status{};
  s = set();
  if (s == Status{}) done.fetch_or(bit, std::memory_order_release);
  return s;
}

}  // namespace ff
