// ca_digits.cuh -- the FP64 Gram Y Y^T of sampled rows on the FP16 tensor
// cores, by digit products (the error-free splitting of Ozaki, Ogita,
// Oishi and Rump, Numer. Algorithms 59, 2012, with integer digits and FP32
// accumulation as Mukunoki, Ozaki, Ogita and Imamura, ISC 2020, use it).
//
// A segment of n <= kSeg columns: every row gets one power of two M above its
// largest magnitude there, each element becomes a 55-bit fixed-point integer
// (to nearest, unit 2^-55 M) and the integer seven signed base-256 digits.  A
// digit is exact in FP16; so is every product (in FP32), and the sums of the
// products of digits i and j with one i + j = l stay below 2^24 (l - 1 pairs of
// at most 2^14 over kSeg columns, l <= 6), so the FP32 accumulators of the levels
// l = 2 .. 6 are exact integers.  Levels 7 .. 9 have an accumulator each too,
// rounded in FP32 past 2^24; higher levels are left out.  The levels are put
// together in 64-bit integers and converted once.
//
// What that loses is relative to M_i M_j, not to the entry: the elements' rounding
// at most n 2^-56 (l_i + l_j) M_i M_j, l <= 1 the mean of |y| / M over a row, and the
// rest (0.27 n + 1) 2^-55 M_i M_j (0.02 n up to 160 columns).  FP64 FMAs lose at most n
// 2^-53 S with S = sum |y_ik y_jk|, which for uneven rows is far less.  So an
// entry is formed by digits only where S is known to be large enough for it to
// be within 1.2 max(n, 128) 2^-53 S; the other entries are summed in FP64.
//  - With t the mean of min(|y| / M, 1/8) over a row, in eighths: l <= t, S >= n M_i M_j
//    (t_i + t_j - 1) / 64, as a b >= (a + b - 1/8) / 8 for a, b <= 1/8, and S >= n M^2
//    t^2 / 64 on the diagonal.  So the two smallest t of a segment, summed with the
//    first conversion, clear all its entries if they add up to 1.07 + 0.1 / n, the
//    smaller at least 0.3.  A row of normal numbers has t = 0.8 (largest magnitude 2
//    to 4 times the deviation) or 0.63 (4 to 8 times): with a line at 1.17 four of
//    the 9408 segments of 32 x 8190 in 64 steps were not cleared, 40 us of 1.13 ms;
//    with this one next to none.  A row of zeros loses nothing.
//  - Any other segment starts again with one more product of the same form, of the
//    elements' leading seven bits rounded down (exact integers: S' 2^-14 M_i M_j <=
//    S), and an entry goes by S' >= 42 min(n, 128), that is S >= 0.0026 min(n, 128) M_i M_j
//    (128 x 24001: exponentially distributed 107 us; four fifths zeros 416;
//    elements of 24 decades, next to every entry by FP64, 500, where FP64 tiles of 64 x 64
//    took 557; normal numbers, all cleared, 82).  Rows with an infinity, a NaN or a
//    magnitude outside 2^-480 .. 2^490 fail with every other row.
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

// threadIdx.x as a value of its own: what is derived from it is formed anew and
// not kept over the steps of a solve in registers that then spill (2003 x 24001,
// s b = 128: 1.90 ms a solve, so 1.87).
__device__ __forceinline__ int fresh_tid() {
  int t = (int)threadIdx.x;
  asm volatile("" : "+r"(t));
  return t;
}

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

constexpr int kPitch = 33;  // doubles a row of the tile of sum_listed
// where the entries to sum in FP64 are listed (i * SBP + j each): behind that tile
template <int SBP>
constexpr int kListAt = SBP * kPitch * 8;

// n listed entries over columns [k0, k1) by FP64 FMAs, each added to (add) or
// stored at its place part[row j * sbp + row i] (rows from 64 on: + hi, below: +
// lo).  A few: a warp an entry.  Many: a thread an entry, eight at a time, from
// tiles of 32 columns in shared memory (mem); bound by the FP64 pipe.
template <int SBP>
__device__ __forceinline__ void sum_listed(const double* __restrict__ A, const long long* off,
                                           int sb, long long k0, long long k1, int n, bool add,
                                           unsigned char* mem, double* __restrict__ part, int sbp,
                                           int lo, int hi) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint16_t* lst = reinterpret_cast<const uint16_t*>(mem + kListAt<SBP>);
  auto store = [&](int i, int j, double s) {
    double* at = part + (long long)(j + (j < 64 ? lo : hi)) * sbp + i + (i < 64 ? lo : hi);
    *at = add ? *at + s : s;
  };
  if (n <= 64) {
    for (int e = warp; e < n; e += 8) {
      const int i = lst[e] / SBP, j = lst[e] % SBP;
      double x[kSeg / 32], y[kSeg / 32], s = 0.0;
#pragma unroll
      for (int q = 0; q < kSeg / 32; ++q) {
        const long long k = min(k0 + 32 * q + lane, k1 - 1);
        x[q] = __ldg(A + off[i] + k);
        y[q] = __ldg(A + off[j] + k);
      }
#pragma unroll
      for (int q = 0; q < kSeg / 32; ++q)
        if (k0 + 32 * q + lane < k1) s = fma(x[q], y[q], s);
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) store(i, j, s);
    }
    return;
  }
  constexpr int Q = 8;
  double* tile = reinterpret_cast<double*>(mem);
  for (int e0 = 0; e0 < n; e0 += 256 * Q) {
    int ti[Q], tj[Q];
    double s[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int c = lst[min(e0 + tid + 256 * q, n - 1)];
      ti[q] = c / SBP * kPitch;
      tj[q] = c % SBP * kPitch;
      s[q] = 0.0;
    }
    for (long long k = k0; k < k1; k += 32) {
      main_sync();
#pragma unroll 4
      for (int r = warp; r < sb; r += 8) {
        const double x = __ldg(A + off[r] + min(k + lane, k1 - 1));
        tile[r * kPitch + lane] = k + lane < k1 ? x : 0.0;
      }
      main_sync();
      for (int c = 0; c < 32; ++c)
#pragma unroll
        for (int q = 0; q < Q; ++q)
          if (e0 + 256 * q < n) s[q] = fma(tile[ti[q] + c], tile[tj[q] + c], s[q]);
    }
#pragma unroll
    for (int q = 0; q < Q; ++q)
      if (e0 + tid + 256 * q < n) store(ti[q] / kPitch, tj[q] / kPitch, s[q]);
  }
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

  unsigned char* dig;   // 1024-byte aligned digits of two stages; after the passes the
                        // entries to sum in FP64 (a list) and their columns (a tile)
  uint64_t* bars;       // [0], [1]: stage buffer read by the MMAs; [2]: all MMAs of a
                        // pass; [3], [4]: stage buffer converted (a warp each)
  uint32_t* cmd;        // [2]: what the MMA warp does with each buffer
  uint32_t tmem;
  int* emax;            // [SBP] largest biased exponent of each row
  float* wt;            // [SBP] 1, 0 (a row of zeros) or infinity (not for digits)
  int* nlist;           // entries to sum in FP64
  uint32_t* tmin;       // [16] each warp's two smallest t n
  int64_t* diag;        // [SBP] (SBP = 128)
  int tid0 = 0;         // fresh_tid() of the segment
  uint32_t gt = 0;      // stages so far (buffers and phases run on)
  uint32_t ph = 0;      // passes so far
  // gram<true>: two groups of 64 rows of a larger Gram, at rows and columns lo
  // and hi + 64 of the partial; the diagonal block of a group only if owned
  int lo = 0, hi = 0;
  bool own_lo = true, own_hi = true;
  __device__ __forceinline__ bool owned(int i, int j) const {  // i >= j
    return i >= 64 ? (j < 64 || own_hi) : own_lo;
  }

  static_assert(kListAt<SBP> + SBP * (SBP + 1) <= 2 * kStage, "tile and list fit there");
  __device__ __forceinline__ uint16_t* list() const {
    return reinterpret_cast<uint16_t*>(dig + kListAt<SBP>);
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
    const long long kk = k + 2 * (tid0 & 15);
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
  // one stage of 32 columns: digits 1 .. ND of every row (ND = 0: the leading
  // seven bits of its magnitudes, in the place of digit 1); SUM: min(|y| / M, 1/8) in
  // units of 2^-23 added to ts
  template <int ND, bool SUM>
  __device__ __forceinline__ void convert(const Rows& rw, const double (&x)[kRows][2],
                                          unsigned char* buf, uint32_t (&ts)[kRows]) const {
    const int warp = tid0 >> 5, lane = tid0 & 31, l = lane & 15;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int r = 2 * (warp + 8 * i) + (lane >> 4);
      uint32_t hi[2], lo[2], qh[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const uint64_t u = (uint64_t)__double_as_longlong(x[i][e]);
        const int ex = (int)(u >> 52) & 0x7ff;
        const uint64_t m = ((u & 0xfffffffffffffull) | ((uint64_t)(ex != 0) << 52)) << 2;
        const int sh = min(rw.em[i] - (ex ? ex : 1), 63);  // >= 0
        const uint64_t q = (m + ((1ull << sh) >> 1)) >> sh;
        const uint64_t t = ((int64_t)u < 0 ? (uint64_t)0 - q : q) + 0x0080808080808080ull;
        qh[e] = (uint32_t)(q >> 32);
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
      const uint32_t head = __byte_perm(qh[0], qh[1], 0x7632u);  // (0 .. 128: q <= 2^55)
      if constexpr (ND == 0)
        *reinterpret_cast<uint32_t*>(buf + at) = h2_sub(head | 0x64006400u, 0x64006400u);
      if constexpr (SUM) ts[i] += min(qh[0], 1u << 20) + min(qh[1], 1u << 20);
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
        if ((c & 3u) == 3u) {
          issue<2, 2>(buf, nb, first, half);  // (S': one product, as level 2)
        } else if constexpr (SBP <= 64) {
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

  // one pass over the segment: levels L0 .. L1 (L1 = 1: S') into tensor memory,
  // with SUM ts too; landed() returns once the products are there
  template <int L0, int L1, bool SUM = false>
  __device__ bool pass(const double* __restrict__ A, const Rows& rw, int sb, long long k0,
                       long long k1, unsigned* err, bool ok, uint32_t (&ts)[kRows]) {
    const int nb = (sb + 15) & ~15;
    double x[kRows][2];
    load(A, rw, k0, k1, x);
    for (long long k = k0; k < k1; k += 32, ++gt) {
      const uint32_t bi = gt & 1;
      unsigned char* buf = dig + bi * kStage;
      if (gt >= 2 && ok) ok = mbar_wait_grid(&bars[bi], ((gt >> 1) - 1) & 1, err);
      convert<(L1 - 1 < kDigits ? L1 - 1 : kDigits), SUM>(rw, x, buf, ts);
      load(A, rw, k + 32, k1, x);  // (lands while the MMAs of this stage run)
      if (tid0 == 0)
        cmd[bi] = (uint32_t)(L1 == 1 ? 3 : L0 == 6 ? 2 : L1 == 5 ? 1 : 0) | (k == k0 ? kFirst : 0u) |
                  (k + 32 >= k1 ? kLast : 0u) | (k + 16 >= k1 ? kHalf : 0u) | (uint32_t)nb << 8;
      fence_proxy_async_smem();
      tc_fence_before();
      __syncwarp();
      if ((tid0 & 31) == 0) mbar_arrive(&bars[3 + bi]);
    }
    return ok;
  }
  __device__ __forceinline__ bool landed(unsigned* err, bool ok) {
    if (ok) ok = mbar_wait_grid(&bars[2], ph & 1, err);
    ++ph;
    tc_fence_after();
    return ok;
  }

  // Whether the two smallest t of the segment's sb rows let every entry be formed
  // by digits (all main warps; ts from the conversion).
  __device__ __forceinline__ bool even(const uint32_t (&ts)[kRows], int sb, uint32_t n) const {
    const int warp = tid0 >> 5, lane = tid0 & 31;
    constexpr uint32_t kNone = 0x3fffffffu;
    uint32_t t1 = kNone, t2 = kNone;
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      uint32_t t = ts[i];
#pragma unroll
      for (int o = 8; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      const int r = 2 * (warp + 8 * i) + (lane >> 4);
      if (r >= sb || wt[min(r, sb - 1)] == 0.f) t = kNone;
      t2 = min(t2, max(t1, t));
      t1 = min(t1, t);
    }
    {
      const uint32_t o1 = __shfl_xor_sync(0xffffffffu, t1, 16);
      const uint32_t o2 = __shfl_xor_sync(0xffffffffu, t2, 16);
      t2 = min(max(t1, o1), min(t2, o2));
      t1 = min(t1, o1);
    }
    if (lane < 2) tmin[2 * warp + lane] = lane == 0 ? t1 : t2;
    main_sync();
    t2 = lane < 16 ? tmin[lane] : kNone;
    t1 = __reduce_min_sync(0xffffffffu, t2);
    if (__popc(__ballot_sync(0xffffffffu, t2 == t1)) > 1) t2 = t1;
    else t2 = __reduce_min_sync(0xffffffffu, t2 == t1 ? kNone : t2);
    // t n in units of 2^-20: t1 + t2 >= 1.07 + 0.1 / n, t1 >= 0.3
    return t1 + t2 >= 1121977u * n + 104858u && t1 >= 314573u * n;
  }

  // The passes of a segment whose emax and wt stand, and its entries into part; false,
  // with nothing stored, if the rows are not even.  UNEVEN: S' first, and the
  // entries that it does not clear summed in FP64.
  template <bool PAIR, bool UNEVEN>
  __device__ __forceinline__ bool passes(const double* __restrict__ A, const long long* off, int sb,
                                         long long k0, long long k1, double* __restrict__ part,
                                         int sbp, bool add, unsigned* err, bool& ok) {
    const int tid = tid0, warp = tid >> 5, lane = tid & 31;
    auto at_ = [&](int r) { return PAIR ? r + (r < 64 ? lo : hi) : r; };  // a row's place in part
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
    uint32_t ts[kRows] = {};
    // chunks of 16 columns, shared by the two warps of a lane quadrant
    uint64_t plain = 0;  // the entries of this thread's chunks to sum in FP64, sixteen bits each
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
      [[maybe_unused]] const uint32_t pl = (uint32_t)(plain >> (cc >> 5 << 4));
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int j = cc + q;
        if (j > row) break;
        if constexpr (UNEVEN) {
          if (pl >> q & 1u) {
            list()[atomicAdd(nlist, 1)] = (uint16_t)(row * SBP + j);
            continue;
          }
        }
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
    if constexpr (UNEVEN) {
      if (tid == 0) *nlist = 0;
      ok = landed(err, pass<2, 1>(A, rw, sb, k0, k1, err, ok, ts));
      const float line = 42.f * (float)min(k1 - k0, 128LL);  // 0.0026 2^14
      chunks([&](int cc) {
        uint32_t x[16];
        tmem_ld16(tbase + (uint32_t)cc, x);
        if (row >= sb) return;
        const float lr = line * wt[row];
        uint32_t pl = 0;
#pragma unroll
        for (int q = 0; q < 16; ++q)  // (a row of zeros and an infinite weight: a NaN, not >=)
          pl |= !(__uint_as_float(x[q]) >= lr * wt[min(cc + q, row)]) ? 1u << q : 0u;
        plain |= (uint64_t)pl << (cc >> 5 << 4);
      });
      tc_fence_before();
      main_sync();
    }
    if constexpr (SBP <= 64) {
      ok = pass<2, 9, !UNEVEN>(A, rw, sb, k0, k1, err, ok, ts);
      const bool go = UNEVEN || even(ts, sb, (uint32_t)(k1 - k0));
      ok = landed(err, ok);
      if (!go) return false;
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
      ok = pass<2, 5, !UNEVEN>(A, rw, sb, k0, k1, err, ok, ts);
      const bool go = UNEVEN || even(ts, sb, (uint32_t)(k1 - k0));
      ok = landed(err, ok);
      if (!go) return false;
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
      ok = landed(err, pass<6, 9>(A, rw, sb, k0, k1, err, ok, ts));
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
    if constexpr (!UNEVEN) {
      main_sync();  // the accumulators are read
    } else if (!main_any(!ok) && *nlist > 0) {
      // (the list is complete; with a wait given up, digits written late might
      // have taken its place, and nothing is summed)
      sum_listed<SBP>(A, off, sb, k0, k1, *nlist, add, dig, part, sbp, PAIR ? lo : 0,
                      PAIR ? hi : 0);
      main_sync();  // (the digits' memory, the list and its length are free again)
    }
    return true;
  }
  // (a function of its own, on a copy: inlined, its registers cost the loops of
  // the other segments 20 us of 1.1 ms, X^T 1500 x 8190, s b = 32)
  struct After {
    uint32_t gt, ph;
    bool ok;
  };
  template <bool PAIR>
  static __device__ __noinline__ After passes_uneven(DigitGram dg, const double* __restrict__ A,
                                                     const long long* off, int sb, long long k0,
                                                     long long k1, double* __restrict__ part,
                                                     int sbp, bool add, unsigned* err, bool ok) {
    dg.template passes<PAIR, true>(A, off, sb, k0, k1, part, sbp, add, err, ok);
    return After{dg.gt, dg.ph, ok};
  }

  // Gram of rows off[0 .. sb) over columns [k0, k1), added to (add) or stored
  // in part[j * sbp + i], i >= j.  All 256 threads; false once a wait gave up.
  template <bool PAIR = false>
  __device__ bool gram(const double* __restrict__ A, const long long* off, int sb, long long k0,
                       long long k1, double* __restrict__ part, int sbp, bool add, unsigned* err,
                       bool ok) {
    tid0 = fresh_tid();
    const int warp = tid0 >> 5, lane = tid0 & 31;
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
        bool zero = false;
        if (e == 0) {  // zeros (or subnormal numbers only: not for digits)
          bool nz = false;
          for (long long k = k0 + lane; k < k1; k += 32) nz |= __ldg(A + off[r] + k) != 0.0;
          zero = !__any_sync(0xffffffffu, nz);
          e = zero ? 1023 : 1;
        }
        const bool out = e < 543 || e > 1513;
        plain |= out;
        if (lane == 0) {
          emax[r] = e;
          wt[r] = zero ? 0.f : out ? __int_as_float(0x7f800000) : 1.f;
        }
      }
    }
    if (!main_any(plain) && passes<PAIR, false>(A, off, sb, k0, k1, part, sbp, add, err, ok))
      return ok;
    const After u = passes_uneven<PAIR>(*this, A, off, sb, k0, k1, part, sbp, add, err, ok);
    gt = u.gt;
    ph = u.ph;
    return u.ok;
  }
};

}  // namespace
