// Checks of the plan of the persistent launches (paper_1612_04003_gb300/csrc/
// ca_steps_plan.h): runs of outer steps cover a solve's full steps in order, end
// at every host decision and before a short last step, and are short enough
// for a grid's 32-bit counts.  Prints "ALL OK".
#include <cstdio>
#include <cstdlib>

#include "ca_steps_plan.h"

static int fails = 0;
#define CHECK(c)                                              \
  do {                                                        \
    if (!(c)) {                                               \
      std::printf("FAIL %s:%d %s\n", __FILE__, __LINE__, #c); \
      ++fails;                                                \
    }                                                         \
  } while (0)

static void check_runs(long long s, long long H, long long every) {
  const long long full = H / s;  // steps of s blocks
  auto boundary = [&](long long j) { return every > 0 && (j + 1) % every == 0; };
  long long k = 0;
  while (k < full) {
    const long long k1 = casteps::run_end(k, s, H, boundary);
    CHECK(k1 > k && k1 <= full);
    CHECK((k1 - k) * 1024 < (1LL << 31));  // counts of a grid of up to 1024 CTAs
    for (long long j = k; j + 1 < k1 && every > 0; ++j) CHECK(!boundary(j));
    if (k1 <= k) break;
    k = k1;
  }
  CHECK(k == full);
}

int main() {
  check_runs(1, 200, 0);
  check_runs(8, 129, 8);
  check_runs(16, 4096, 3);
  check_runs(4, 1, 0);
  check_runs(1, 50000000, 0);  // would wrap the counts in one launch
  check_runs(3, 100000001, 0);
  check_runs(2, 300000, 100000);
  if (fails == 0) std::printf("ALL OK\n");
  return fails != 0;
}
