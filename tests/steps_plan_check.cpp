// Checks of the plan of the persistent launches (paper_1612_04003_gb300/csrc/
// ca_steps_plan.h): runs of outer steps cover a solve's full steps in order, end
// at every host decision and before a short last step, and are short enough
// for a grid's 32-bit counts; the column CTAs of the FP64 launch leave room for the
// others, have columns each, and no more work a step than the bounded waits
// allow.  Prints "ALL OK".
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

static void check_columns(int b, int s, long long K, int sms) {
  const int P = casteps::persist64_columns(b, s, K, sms);
  CHECK(P >= 0);
  if (b > 16 || s * b > 128) CHECK(P == 0);
  if (P == 0) return;
  CHECK(P + 1 + (s < casteps::kMaxInv ? s : casteps::kMaxInv) <= sms);
  CHECK((K + 15) / 16 >= P);  // a share of at least 16 columns each
  // a step of FP64 FMAs alone (the pipe does two a clock) at 1 GHz, five times over,
  // stays below the 2 s of a wait
  const double cols = (double)((K + P - 1) / P), sb = (double)s * b;
  CHECK(5.0 * cols * (sb * (sb + 1) / 2 + 2 * sb) / 2 / 1e9 < 2.0);
}

int main() {
  for (int sms : {1, 2, 18, 76, 152})
    for (int b : {1, 3, 8, 16, 17})
      for (int s : {1, 4, 16, 42, 128})
        for (long long K = 1; K < 40000000000LL; K = K * 3 + 7) check_columns(b, s, K, sms);
  CHECK(casteps::persist64_columns(8, 4, 8190, 152) == 147);
  CHECK(casteps::persist64_columns(4, 1, 1024, 152) == 32);
  CHECK(casteps::persist64_columns(16, 8, 24001, 152) == 143);
  CHECK(casteps::persist64_columns(16, 8, 200000000, 152) == 0);  // 205 GB at 128 rows
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
