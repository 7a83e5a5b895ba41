// Plan of the persistent launches, which run consecutive outer steps of a dense
// solve (Algorithms 2 and 4) in one grid (host only, no CUDA).
#pragma once

#include <algorithm>

namespace casteps {

// Outer steps of one launch: a grid's counts go up to its CTAs times its steps
// and are compared as 32-bit numbers (152 x 65536 = 10^7; past 2^32 / 152 = 28 M
// steps they would wrap).  A new launch costs a few steps' time.
constexpr long long kMaxRun = 65536;

// End of the run of outer steps that starts at step k: at most kMaxRun steps, all
// of s blocks (of H in all), and up to the first one that boundary(step) follows
// (a host decision: a check, a due recomputation).
template <typename Boundary>
long long run_end(long long k, long long s, long long H, Boundary&& boundary) {
  const long long n_outer = (H + s - 1) / s;
  long long k1 = k + 1;
  while (k1 < n_outer && k1 - k < kMaxRun && s * (k1 + 1) <= H && !boundary(k1 - 1)) ++k1;
  return k1;
}

}  // namespace casteps
