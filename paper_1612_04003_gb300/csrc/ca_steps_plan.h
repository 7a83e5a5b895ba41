// Plan of the persistent launches, which run consecutive outer steps of a dense
// solve (Algorithms 2 and 4) in one grid (host only, no CUDA).
#pragma once

#include <algorithm>

namespace casteps {

// Outer steps of one launch: a grid's counts go up to its CTAs times its steps
// and are compared as 32-bit numbers (152 x 65536 = 10^7; past 2^32 / 152 = 28 M
// steps they would wrap).  A new launch costs a few steps' time.
constexpr long long kMaxRun = 65536;

constexpr int kMaxInv = 16;  // inverse CTAs of the FP64 launch

// Column CTAs of the persistent FP64 launch for s blocks of b rows a step over K
// columns: every SM but the inverse CTAs' and the chain's, with at least 32
// columns each.  0: the launches per step instead, for what it does not cover
// (b > 16, s b > 128) and where a step is so long that a wait for the slowest CTA
// could reach the limit of its bounded waits (2 s): 2^29 FP64 FMAs a CTA, 0.15 s of
// its SM's FP64 pipe (128 rows: 8.6 M columns), as many as a step takes whose
// entries are all summed in FP64.  Launches are no part of such a step's time
// (128 rows, 8 M columns: 27 ms at least).
inline int persist64_columns(int b, int s, long long K, int num_sms) {
  if (b > 16 || s * b > 128) return 0;
  const long long sb = (long long)s * b;
  const long long P = std::min<long long>(num_sms - 1 - std::min(s, kMaxInv), (K + 31) / 32);
  if (P <= 0) return 0;
  const long long fmas = ((K + P - 1) / P) * (sb * (sb + 1) / 2 + 2 * sb);
  return fmas <= (1LL << 29) ? (int)P : 0;
}

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
