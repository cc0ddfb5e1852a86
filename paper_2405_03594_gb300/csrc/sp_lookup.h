// sp_lookup.h -- a positive number that is looked up at its first use and kept.  Host only.
#pragma once

#include <atomic>

namespace sp {

// The kept number, or what `lookup` gives now.  A lookup that fails (0 or less) is not kept: its cause
// may pass, and the next call asks again.
template <class F>
int kept_or_looked_up(std::atomic<int>& kept, F lookup) {
  int n = kept.load(std::memory_order_acquire);
  if (n > 0) return n;
  n = lookup();
  if (n > 0) kept.store(n, std::memory_order_release);
  return n > 0 ? n : 0;
}

}  // namespace sp
