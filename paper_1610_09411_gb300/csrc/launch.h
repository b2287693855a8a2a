// launch.h -- grids of the persistent kernels (plain C++).
#pragma once
#include <algorithm>
#include <cstdint>

namespace esc {

// CTAs of `threads` threads for `items` work items: as many as fit the device at
// once (`fit` per SM), no more than cta_per_sm CTAs of 512 threads or their equal
// per SM when the caller set that (0: not set), at most one per item.
inline unsigned persistent_grid(int fit, int threads, int cta_per_sm, int sms, int64_t items) {
  int per_sm = std::max(1, fit);
  if (cta_per_sm > 0) per_sm = std::min(per_sm, std::max(1, cta_per_sm * 512 / threads));
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)per_sm * sms, items));
}

}  // namespace esc
