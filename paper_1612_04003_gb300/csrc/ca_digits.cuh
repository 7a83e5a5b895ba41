// ca_digits.cuh -- the FP64 Gram Y Y^T of sampled rows on the FP16 tensor
// cores, by exact digit products (the error-free splitting of Ozaki, Ogita,
// Oishi and Rump, Numer. Algorithms 59, 2012, with integer digits and FP32
// accumulation as Mukunoki, Ozaki, Ogita and Imamura, ISC 2020, use it).
//
// A segment of at most kSeg columns: every row gets one power of two above its
// largest magnitude there, each element becomes a 55-bit fixed-point integer
// (to nearest) and the integer seven signed base-256 digits.  A digit is exact
// in FP16; so is every product (in FP32), and the sums of the products of digits i and
// j with one i + j = l stay below 2^24 (l - 1 pairs of at most 2^14 over kSeg
// columns, l <= 6), so the FP32 accumulators of the levels l = 2 .. 6 are
// exact integers.  Levels 7 .. 9 share one accumulator (their FP32 rounding is
// below 2^-54 of the product of the two rows' largest magnitudes); higher
// levels are below that and left out.  The levels are put together in 64-bit
// integers and converted once.  Rows with an infinity, a NaN or a magnitude
// outside 2^-480 .. 2^490 take the plain FP64 sums instead.
//
// Why: the FP64 pipe does two FMAs a clock and SM (1.25 TFLOP/s).  The 34
// digit products of a 128-row tile and 32 columns take ~4,400 cycles of the
// tensor pipe where 128 x 129 / 2 x 32 FMAs take 132,000 of the FP64 pipe.
#pragma once
#include "ca_common.cuh"
#include "ca_tc.cuh"

namespace {

constexpr int kSeg = 192;  // columns whose level sums stay exact in FP32
constexpr int kDigits = 7;

// Named barrier 1 over the eight warps that form a Gram partial (a CTA may have
// others), and the same with a vote.
__device__ __forceinline__ void main_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ bool main_any(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbarrier.cta.red.or.pred q, 1, 256, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ uint32_t h2_sub(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// v 2^e, rounded to nearest, on the integer pipe (a conversion of the FP64
// pipe holds a scheduler for 64 cycles); the result is a normal number.
__device__ __forceinline__ double fixed_to_double(int64_t v, int e) {
  uint64_t m = v < 0 ? (uint64_t)0 - (uint64_t)v : (uint64_t)v;
  int lz = __clzll((long long)m);
  m <<= lz & 63;
  uint64_t t = m + 0x400u;
  if (t < m) {  // rounded up to the next power of two
    t = 1ull << 63;
    --lz;
  }
  const uint64_t b = ((uint64_t)(uint32_t)(1086 - lz + e) << 52) | ((t >> 11) & 0xfffffffffffffull) |
                     ((uint64_t)v & (1ull << 63));
  return v == 0 ? 0.0 : __longlong_as_double((long long)b);
}

// SBP rows (32, 64 or 128), the eight main warps of a CTA.  Tensor memory: one
// accumulator of SBP columns a level.  SBP = 128 holds four of the eight at
// once: levels 2 .. 5, then (the columns converted again) levels 6 .. 9.
template <int SBP>
struct DigitGram {
  static constexpr int kSlice = SBP * 64;              // 32 FP16 digits a row
  static constexpr int kStage = kDigits * kSlice;
  // the M = 128 MMA reads 128 rows of a slice: slack behind the last one
  static constexpr int kSmem = 2 * kStage + (128 - (SBP < 128 ? SBP : 128)) * 64 + 1024;
  static constexpr int kTmemCols = SBP == 32 ? 256 : 512;

  unsigned char* dig;   // 1024-byte aligned digits of two stages
  uint64_t* bars;       // [0], [1]: stage buffer read by the MMAs; [2]: all MMAs of a
                        // pass; [3], [4]: stage buffer converted (a warp each)
  uint32_t* cmd;        // [2]: what the MMA warp does with each buffer
  uint32_t tmem;
  int* emax;            // [SBP] largest biased exponent of each row
  int64_t* diag;        // [SBP] (SBP = 128)
  uint32_t gt = 0;      // stages so far (buffers and phases run on)
  uint32_t ph = 0;      // passes so far
  // gram<true>: two groups of 64 rows of a larger Gram, at rows and columns lo
  // and hi + 64 of the partial; the diagonal block of a group only if owned
  int lo = 0, hi = 0;
  bool own_lo = true, own_hi = true;
  __device__ __forceinline__ bool owned(int i, int j) const {  // i >= j
    return i >= 64 ? (j < 64 || own_hi) : own_lo;
  }

  // This thread's rows 2 (warp + 8 i) + lane / 16, columns 2 (lane % 16) and
  // the next of a stage.
  static constexpr int kRows = SBP / 16;
  struct Rows {
    long long off[kRows];  // (rows past sb: the last row again, never stored)
    int em[kRows];
  };
  // (unconditional loads at clamped columns, then a select: a condition on
  // each load makes branches that wait for one load after another)
  __device__ __forceinline__ void load(const double* __restrict__ A, const Rows& rw, long long k,
                                       long long k1, double (&x)[kRows][2]) const {
    const long long kk = k + 2 * (threadIdx.x & 15);
    const long long ka = min(kk, k1 - 1), kb = min(kk + 1, k1 - 1);
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      x[i][0] = __ldg(A + rw.off[i] + ka);
      x[i][1] = __ldg(A + rw.off[i] + kb);
    }
    if (kk + 1 >= k1) {
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        x[i][1] = 0.0;
        if (kk >= k1) x[i][0] = 0.0;
      }
    }
  }
  // one stage of 32 columns: digits 1 .. ND of every row (rows past sb: zero)
  template <int ND>
  __device__ __forceinline__ void convert(const Rows& rw, const double (&x)[kRows][2],
                                          unsigned char* buf) const {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane & 15;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int r = 2 * (warp + 8 * i) + (lane >> 4);
      uint32_t hi[2], lo[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint64_t u = (uint64_t)__double_as_longlong(x[i][e]);
        const int ex = (int)(u >> 52) & 0x7ff;
        const uint64_t m = ((u & 0xfffffffffffffull) | ((uint64_t)(ex != 0) << 52)) << 2;
        const int sh = min(rw.em[i] - (ex ? ex : 1), 63);  // >= 0
        const uint64_t q = (m + ((1ull << sh) >> 1)) >> sh;
        const uint64_t t = ((int64_t)u < 0 ? (uint64_t)0 - q : q) + 0x0080808080808080ull;
        hi[e] = (uint32_t)(t >> 32);
        lo[e] = (uint32_t)t;
      }
      const uint32_t at = (uint32_t)((r >> 3) * 512 + (r & 7) * 64 +
                                     (((l >> 2) ^ ((r >> 1) & 3)) << 4) + (l & 3) * 4);
#pragma unroll
      for (int d = 0; d < ND; ++d) {  // digit d + 1 of both columns
        // byte 6 - d of the two (the first digit has nine bits) under the FP16
        // exponent of 1024, less 1024 + 128
        const uint32_t w0 = d < 3 ? hi[0] : lo[0], w1 = d < 3 ? hi[1] : lo[1];
        const uint32_t sel = d == 0 ? 0x7632u : d == 1 ? 0x0501u : d == 2 ? 0x0400u
                             : d == 3 ? 0x0703u : d == 4 ? 0x0602u : d == 5 ? 0x0501u : 0x0400u;
        const uint32_t f = (__byte_perm(w0, w1, sel) & (d == 0 ? 0x01ff01ffu : 0x00ff00ffu)) | 0x64006400u;
        *reinterpret_cast<uint32_t*>(buf + d * kSlice + at) = h2_sub(f, 0x64806480u);
      }
    }
  }

  // MMAs of one stage: pairs (i, j) of digits with level i + j in [L0, L1],
  // level l into accumulator l - L0
  template <int L0, int L1>
  __device__ __forceinline__ void issue(uint32_t buf, int nb, bool first, bool half) const {
    const uint32_t id = idesc_f16(128, nb);
    const uint64_t base = sw64_kmajor_desc(buf);  // (the address field is in 16-byte units)
#pragma unroll
    for (int l = L0; l <= L1; ++l) {
      const uint32_t d = tmem + (uint32_t)(SBP * (l - L0));
#pragma unroll
      for (int i = 1; i <= kDigits; ++i) {
        const int j = l - i;
        if (j < 1 || j > kDigits) continue;
        const bool start = i == (l > 8 ? l - kDigits : 1);
#pragma unroll
        for (int kk = 0; kk < 2; ++kk)
          if (kk == 0 || !half)
            mma_bf16(d, base + (uint32_t)(((i - 1) * kSlice + kk * 32) >> 4),
                     base + (uint32_t)(((j - 1) * kSlice + kk * 32) >> 4), id,
                     start && kk == 0 ? (first ? 0u : 1u) : 1u);
      }
    }
  }

  // The MMA warp (a warp of its own: an issue waits until the tensor pipe takes
  // it, which in a converting warp held the conversion of the next stage):
  // stages in order until stop().
  static constexpr uint32_t kFirst = 16u, kLast = 32u, kStop = 64u, kHalf = 128u;
  __device__ void mma_loop(unsigned* err) const {
    for (uint32_t g = 0;; ++g) {
      const uint32_t bi = g & 1;
      if (!mbar_wait_grid(&bars[3 + bi], (g >> 1) & 1, err)) return;
      const uint32_t c = *(volatile uint32_t*)&cmd[bi];
      if (c & kStop) return;
      tc_fence_after();
      if (elect_one()) {
        const uint32_t buf = smem_u32(dig + bi * kStage);
        const int nb = (int)(c >> 8);
        const bool first = c & kFirst, half = c & kHalf;  // (half: at most 16 columns)
        if constexpr (SBP <= 64) {
          issue<2, 9>(buf, nb, first, half);
        } else {
          if ((c & 3u) == 1u) issue<2, 5>(buf, nb, first, half);
          else issue<6, 9>(buf, nb, first, half);
        }
        mma_commit(&bars[bi]);
        if (c & kLast) mma_commit(&bars[2]);
      }
      __syncwarp();
    }
  }
  // ends mma_loop (every pass so far is complete)
  __device__ void stop() {
    main_sync();
    if (threadIdx.x == 0) {
      cmd[gt & 1] = kStop;
      for (int q = 0; q < 8; ++q) mbar_arrive(&bars[3 + (gt & 1)]);
    }
  }

  // one pass over the segment: levels L0 .. L1 into tensor memory
  template <int L0, int L1>
  __device__ bool pass(const double* __restrict__ A, const Rows& rw, int sb, long long k0,
                       long long k1, unsigned* err, bool ok) {
    const int nb = (sb + 15) & ~15;
    double x[kRows][2];
    load(A, rw, k0, k1, x);
    for (long long k = k0; k < k1; k += 32, ++gt) {
      const uint32_t bi = gt & 1;
      unsigned char* buf = dig + bi * kStage;
      if (gt >= 2 && ok) ok = mbar_wait_grid(&bars[bi], ((gt >> 1) - 1) & 1, err);
      convert<(L1 - 1 < kDigits ? L1 - 1 : kDigits)>(rw, x, buf);
      load(A, rw, k + 32, k1, x);  // (lands while the MMAs of this stage run)
      if (threadIdx.x == 0)
        cmd[bi] = (uint32_t)(L0 == 6 ? 2 : (L1 == 5 ? 1 : 0)) | (k == k0 ? kFirst : 0u) |
                  (k + 32 >= k1 ? kLast : 0u) | (k + 16 >= k1 ? kHalf : 0u) | (uint32_t)nb << 8;
      fence_proxy_async_smem();
      tc_fence_before();
      __syncwarp();
      if ((threadIdx.x & 31) == 0) mbar_arrive(&bars[3 + bi]);
    }
    if (ok) ok = mbar_wait_grid(&bars[2], ph & 1, err);
    ++ph;
    tc_fence_after();
    return ok;
  }

  // Gram of rows off[0 .. sb) over columns [k0, k1), added to (add) or stored
  // in part[j * sbp + i], i >= j.  All 256 threads; false once a wait gave up.
  template <bool PAIR = false>
  __device__ bool gram(const double* __restrict__ A, const long long* off, int sb, long long k0,
                       long long k1, double* __restrict__ part, int sbp, bool add, unsigned* err,
                       bool ok) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    auto at_ = [&](int r) { return PAIR ? r + (r < 64 ? lo : hi) : r; };  // a row's place in part
    // largest exponent of each row in the segment
    bool plain = false;
    constexpr int RB = 4;  // rows in flight a warp
    for (int r0 = warp; r0 < sb; r0 += 8 * RB) {
      uint32_t h[RB];
#pragma unroll
      for (int u = 0; u < RB; ++u) {
        const double* row = A + off[min(r0 + 8 * u, sb - 1)];
        h[u] = 0;
#pragma unroll
        for (int q = 0; q < kSeg / 32; ++q)
          h[u] = max(h[u], __ldg(reinterpret_cast<const uint32_t*>(
                               row + min(k0 + 32 * q + lane, k1 - 1)) + 1) & 0x7fffffffu);
      }
#pragma unroll
      for (int u = 0; u < RB; ++u) {
        const int r = r0 + 8 * u;
        if (r >= sb) break;
        int e = (int)(__reduce_max_sync(0xffffffffu, h[u]) >> 20);
        if (e == 0) {  // zeros (or subnormal numbers only: the plain sums)
          bool nz = false;
          for (long long k = k0 + lane; k < k1; k += 32) nz |= __ldg(A + off[r] + k) != 0.0;
          if (!__any_sync(0xffffffffu, nz)) e = 1023;
        }
        plain |= e < 543 || e > 1513;
        if (lane == 0) emax[r] = e;
      }
    }
    if (main_any(plain)) {
      for (int e = tid; e < sb * (sb + 1) / 2; e += 256) {
        int i, j;
        tri_decode(e, i, j);
        if (PAIR && !owned(i, j)) continue;
        double* at = part + (long long)at_(j) * sbp + at_(i);
        double s = add ? *at : 0.0;
        for (long long k = k0; k < k1; ++k) s = fma(__ldg(A + off[i] + k), __ldg(A + off[j] + k), s);
        *at = s;
      }
      main_sync();
      return ok;
    }
    Rows rw;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int r = 2 * (warp + 8 * i) + (lane >> 4);
      rw.off[i] = off[min(r, sb - 1)];
      rw.em[i] = emax[min(r, sb - 1)];
    }
    // warp w: tensor-memory lanes (rows) 32 (w % 4) .. + 31, column chunks of
    // parity w / 4
    const int row = (warp & 3) * 32 + lane;
    const uint32_t tbase = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    const bool act = (warp & 3) * 32 < sb;  // (rows past sb hold garbage)
    // chunks of 16 columns, shared by the two warps of a lane quadrant
    // levels 7 .. 9 of a chunk, in units of level 7
    auto lows = [&](int a, int cc, float (&low)[16]) {
      uint32_t x[16];
      tmem_ld16(tbase + (uint32_t)(SBP * a + cc), x);
#pragma unroll
      for (int q = 0; q < 16; ++q) low[q] = __uint_as_float(x[q]);
      tmem_ld16(tbase + (uint32_t)(SBP * (a + 1) + cc), x);
#pragma unroll
      for (int q = 0; q < 16; ++q) low[q] = fmaf(__uint_as_float(x[q]), 0x1p-8f, low[q]);
      tmem_ld16(tbase + (uint32_t)(SBP * (a + 2) + cc), x);
#pragma unroll
      for (int q = 0; q < 16; ++q) low[q] = fmaf(__uint_as_float(x[q]), 0x1p-16f, low[q]);
    };
    auto put = [&](int cc, const int64_t (&v)[16], const float (&low)[16]) {
      if (row >= sb) return;
      const int er = emax[row] - 2098;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int j = cc + q;
        if (j > row) break;
        // units of level 7 (2^-40 of level 2), then 2^(er + ej - 2098)
        const double g = fixed_to_double(v[q] * 256 + __float2int_rn(low[q]), er + emax[j]);
        double* at = part + (long long)at_(j) * sbp + at_(row);
        *at = add ? *at + g : g;
      }
    };
    auto level = [&](int a, int cc, int64_t (&v)[16]) {
      uint32_t x[16];
      tmem_ld16(tbase + (uint32_t)(SBP * a + cc), x);
#pragma unroll
      for (int q = 0; q < 16; ++q) v[q] = v[q] * 256 + __float2int_rn(__uint_as_float(x[q]));
    };
    const int ccn = (warp & 3) * 32 + 31;  // last column of the quadrant's triangle
    auto chunks = [&](auto&& f) {
      if (act)
        for (int cc = 16 * (warp >> 2); cc < sb && cc <= ccn; cc += 32)
          if (!PAIR || owned(ccn, cc)) f(cc);
    };
    if constexpr (SBP <= 64) {
      ok = pass<2, 9>(A, rw, sb, k0, k1, err, ok);
      chunks([&](int cc) {
        int64_t v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = 0;
        level(0, cc, v);
        level(1, cc, v);
        level(2, cc, v);
        level(3, cc, v);
        level(4, cc, v);
        float low[16];
        lows(5, cc, low);
        put(cc, v, low);
      });
    } else {
      // the integers of levels 2 .. 5 wait in the half of the partial that holds
      // no entry: (row, j) at [row * sbp + j], j < row, and the diagonal in diag
      int64_t* hold = reinterpret_cast<int64_t*>(part) + (long long)at_(min(row, sb - 1)) * sbp;
      ok = pass<2, 5>(A, rw, sb, k0, k1, err, ok);
      chunks([&](int cc) {
        int64_t v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = 0;
        level(0, cc, v);
        level(1, cc, v);
        level(2, cc, v);
        level(3, cc, v);
        if (row < sb) {
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            if (cc + q < row) hold[at_(cc + q)] = v[q];
            if (cc + q == row) diag[row] = v[q];
          }
        }
      });
      tc_fence_before();
      main_sync();
      ok = pass<6, 9>(A, rw, sb, k0, k1, err, ok);
      chunks([&](int cc) {
        int64_t v[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) v[q] = hold[at_(min(cc + q, SBP - 1))];
#pragma unroll
        for (int q = 0; q < 16; ++q)
          if (cc + q == row) v[q] = diag[row];
        level(0, cc, v);
        float low[16];
        lows(1, cc, low);
        put(cc, v, low);
      });
    }
    tc_fence_before();
    main_sync();  // the accumulators are read
    return ok;
  }
};

}  // namespace
