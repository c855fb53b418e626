// Grid width of kernels whose rows of CTAs stride over tiles (host only, no CUDA).
#pragma once
#include <algorithm>

namespace tnq {

// CTAs per row for `batch` rows that each stride over n_tiles tiles, with `slots` CTAs resident at once: the
// width up to four waves with the least (tiles of a CTA, and one more for its start and end) times the waves,
// the smallest of equals.  For a number of waves the widest grid that fits has the fewest tiles per CTA, so a
// few candidates give what trying every width does (thousands of divisions, 7-18 us of host time per launch).
inline long long best_row_grid(long long n_tiles, long long batch, long long slots) {
  const long long most = std::max<long long>(1, std::min(n_tiles, (4 * slots + batch - 1) / batch));
  long long best = 1, best_cost = (n_tiles + 1) * ((batch + slots - 1) / slots);
  for (long long waves = (batch + slots - 1) / slots;; ++waves) {
    const long long widest = std::min(most, waves * slots / batch);
    const long long tiles = (n_tiles + widest - 1) / widest, gx = (n_tiles + tiles - 1) / tiles;
    const long long cost = (tiles + 1) * ((gx * batch + slots - 1) / slots);
    if (cost < best_cost) best = gx, best_cost = cost;
    if (widest == most) return best;
  }
}

}  // namespace tnq
