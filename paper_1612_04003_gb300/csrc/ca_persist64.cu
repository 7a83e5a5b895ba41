// ca_persist64.cu -- consecutive outer steps of a dense FP64 CA-BCD (Alg. 2) /
// CA-BDCD (Alg. 4) solve in one persistent, cooperative launch.
//
// The Gram of step k+1 needs only the sampled indices, so it is formed and
// reduced while the chain of step k runs; what depends on Delta_k is the
// deferred update of v and the projection p_{k+1} = Y_{k+1} v, one sweep over
// the CTA's own columns.  Grid = P column CTAs + up to 16 inverse CTAs + 1
// chain CTA, all resident (cooperative launch); every wait is bounded and gives
// up once any wait of the grid has.
//   column CTA, step k, main warps: wait Delta_{k-1} -> v -= cU Y_{k-1}^T
//     Delta_{k-1} on its columns, p partial -> count P -> Gram partial of step
//     k+1 -> count G; side warps: all G -> its share of the entries summed (Rs,
//     the diagonal blocks) -> count E (s b >= 32: then all P -> its rows of p
//     -> count Q)
//   inverse CTA, step k:  all E -> its diagonal blocks inverted -> count R
//   chain CTA, step k:    all R and P (or Q) -> p -> the s dependent solves ->
//     Delta_k -> count D
// (an inverse CTA that sums its blocks from the partials itself took 11.5 us
// after the last partial of X^T 1500 x 8190, s b = 32; through E 8.3 us)
// Buffers written ahead (partials, Rs, Ginv) alternate by step parity: the
// buffers of step k+1 were last read for step k-1, whose Delta this CTA has
// seen before it writes them.
//
// Bound by latency at few columns a CTA, by the FP64 conversions of the digits
// and FP64 projections at many.  Against four launches a step and a Gram tile
// of 64 x 64 FP64 products whatever s b (ms a solve): X 64 x 1024, b = 4, 200
// solves: s = 1 1.69 against 11.7 (8 us a step), s = 4 0.62 against 3.13 (12
// us); X^T 1500 x 8190, b = 8, s = 4: 1.12 against 6.84 (17 us); 2003 x 24001,
// b = 16, s = 8: 1.89 against 10.2 (70 us a step between recomputations).
#include <algorithm>
#include <atomic>

#include "ca_digits.cuh"
#include "ca_kernels.cuh"
#include "ca_solve.cuh"
#include "ca_steps_plan.h"

namespace {

using casteps::kMaxInv;

constexpr int kT = 256;      // main threads of a CTA (the Gram pass, the chain)
constexpr int kSide = 96;    // side threads of a column CTA (reduction); twelve warps in all
                             // leave 168 registers a thread
constexpr int kMma = 32;     // and the warp that issues the MMAs of the digit Gram
constexpr int kBarSide = 7;  // named barrier of the side warps
constexpr int kSmemMax = 200 * 1024;  // dynamic shared memory a launch may ask for
// Rows of a step up to which the Gram is formed on CUDA cores, digits above (ms a
// solve, CUDA cores against digits: 16 rows x 1024 columns 0.627 / 0.692, 32
// rows x 8190 columns 1.63 / 1.15).
constexpr int kSmallSB = 16;

// Counts in cnt[].  A fast CTA may form the Gram partial of step p + 1 (and its
// side warps reduce it) before a slow one has done step p, but not that of
// step p + 2, which follows Delta_p: G, E and R count even and odd steps apart,
// each to (p / 2 + 1) times its CTAs.
struct Cnt {
  enum { G = 0, E = 2, R = 4, P = 6, Q = 7, D = 8 };
};
// s b from which the column CTAs' side warps sum p, a row a warp, and not the
// chain CTA (ms a solve, chain CTA against side warps: 4 rows 1.72 / 1.96, 16
// rows 0.643 / 0.647, 32 rows 1.157 / 1.096)
constexpr int kRowsSB = 32;

// thread 0 waits, the main warps follow; false once a wait of the grid gave up
__device__ __forceinline__ bool main_wait(const unsigned* p, unsigned target, unsigned* err, bool ok) {
  bool gone = !ok;
  if (threadIdx.x == 0 && ok) gone = !wait_count(p, target, err);
  return !main_any(gone);
}
__device__ __forceinline__ void main_count(unsigned* p) {
  main_sync();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(p, 1u);
  }
}

// Element offsets of the sampled rows (an index out of range is flagged, and
// row 0 stands in for it).
__device__ __forceinline__ void row_offsets(const int* idx, int sb, long long N, long long lda,
                                            long long* out, unsigned* err) {
  for (int r = threadIdx.x; r < sb; r += kT) {
    const long long gi = idx[r];
    const bool in = gi >= 0 && gi < N;
    if (!in) ca_flag(err, CA_DEV_ERR_ARG);
    out[r] = in ? gi * lda : 0;
  }
}

// Gram partial of sb <= 16 rows over columns [k0, k1) on CUDA cores: the
// FP64 pipe does two FMAs a clock and SM, so only the lower triangle is
// formed.  Warp w takes columns 4 w .. 4 w + 3 of each 32-column tile, lane l
// the entries l, l + 32, ...; the warps' sums meet in shared memory.
// smem: tile [sb][33], then sums [8][entries].
__device__ void gram_small(const double* __restrict__ A, const long long* off, int sb, long long k0,
                           long long k1, double* sm, double* __restrict__ part, int sbp) {
  constexpr int kSlots = kSmallSB * (kSmallSB + 1) / 2 / 32 + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int E = sb * (sb + 1) / 2;
  double* tile = sm;
  double* red = sm + kSmallSB * 33;
  int ij[kSlots];
  double acc[kSlots];
#pragma unroll
  for (int q = 0; q < kSlots; ++q) {
    int i = 0, j = 0;
    if (lane + 32 * q < E) tri_decode(lane + 32 * q, i, j);
    ij[q] = i * 33 | (j * 33) << 16;
    acc[q] = 0.0;
  }
  for (long long kt = k0; kt < k1; kt += 32) {
    main_sync();
    const long long k = kt + lane;
#pragma unroll
    for (int q = 0; q < kSmallSB / 8; ++q) {
      const int r = warp + 8 * q;
      const double x = __ldg(A + off[min(r, sb - 1)] + min(k, k1 - 1));
      if (r < sb) tile[r * 33 + lane] = k < k1 ? x : 0.0;
    }
    main_sync();
#pragma unroll
    for (int q = 0; q < kSlots; ++q) {
      if (32 * q < E) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          acc[q] = fma(tile[(ij[q] & 0xffff) + 4 * warp + c], tile[(ij[q] >> 16) + 4 * warp + c], acc[q]);
      }
    }
  }
  main_sync();
#pragma unroll
  for (int q = 0; q < kSlots; ++q)
    if (lane + 32 * q < E) red[warp * E + lane + 32 * q] = acc[q];
  main_sync();
  for (int e = threadIdx.x; e < E; e += kT) {
    double s = red[e];
#pragma unroll
    for (int w = 1; w < 8; ++w) s += red[w * E + e];
    int i, j;
    tri_decode(e, i, j);
    part[(long long)j * sbp + i] = s;
  }
}

// v -= cU Yprev^T Delta (psb > 0) and the projection partial p = Y v of the
// CTA's columns [k0, k1), FP64.  A warp takes four columns at a time (lane =
// 4 row group + column, rows g, g + 8, ...): the eight row groups' sums of a
// column meet by three shuffles, no exchange between warps until the end, and
// the next four columns load while these are summed.  Bound by the FP64 pipe
// (2 FMAs a clock and SM): 2 s b K / (2 P) clocks.
// red: 8 x 8 RQ.
template <int RQ>
__device__ void update_project(const Persist64Args& a, const long long* off, const long long* poff,
                               const double* sdl, int sb, int psb, long long k0, long long k1,
                               double* red, double* __restrict__ pp) {
  const int tid = fresh_tid(), warp = tid >> 5, lane = tid & 31, g = lane >> 2;
  double pacc[RQ], y[RQ], x[RQ], vk;
#pragma unroll
  for (int q = 0; q < RQ; ++q) pacc[q] = 0.0;
  auto rows = [&](const long long* o, int n, long long k, double (&z)[RQ]) {
    const long long kc = min(k, k1 - 1);  // (unconditional loads, then selects)
#pragma unroll
    for (int q = 0; q < RQ; ++q) z[q] = __ldg(a.A + o[min(g + 8 * q, n - 1)] + kc);
#pragma unroll
    for (int q = 0; q < RQ; ++q)
      if (g + 8 * q >= n || k >= k1) z[q] = 0.0;
  };
  const long long kw = k0 + 4 * warp + (lane & 3);
  if (psb > 0) rows(poff, psb, kw, x);
  vk = kw < k1 ? a.v[kw] : 0.0;
  rows(off, sb, kw, y);
  for (long long k = kw; k - (lane & 3) < k1; k += 32) {
    double vn = vk;
    vk = k + 32 < k1 ? a.v[k + 32] : 0.0;
    if (psb > 0) {
      double u = 0.0;
#pragma unroll
      for (int q = 0; q < RQ; ++q)
        if (8 * q < psb) u = fma(x[q], sdl[g + 8 * q], u);  // (x = 0 past psb)
      rows(poff, psb, k + 32, x);
#pragma unroll
      for (int o = 4; o <= 16; o <<= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
      vn -= a.cU * u;
      if (g == 0 && k < k1) a.v[k] = vn;
    }
#pragma unroll
    for (int q = 0; q < RQ; ++q)
      if (8 * q < sb) pacc[q] = fma(y[q], vn, pacc[q]);
    rows(off, sb, k + 32, y);
  }
  // the four columns' sums of a row, by halving exchanges: lane bit 0 keeps
  // the upper or lower half of the values, bit 1 a quarter
#pragma unroll
  for (int j = 0; j < RQ / 2; ++j) {
    const double keep = (lane & 1) ? pacc[j + RQ / 2] : pacc[j];
    pacc[j] = keep + __shfl_xor_sync(0xffffffffu, (lane & 1) ? pacc[j] : pacc[j + RQ / 2], 1);
  }
#pragma unroll
  for (int j = 0; j < RQ / 4; ++j) {
    const double keep = (lane & 2) ? pacc[j + RQ / 4] : pacc[j];
    pacc[j] = keep + __shfl_xor_sync(0xffffffffu, (lane & 2) ? pacc[j] : pacc[j + RQ / 4], 2);
    red[warp * 8 * RQ + g + 8 * (j + (lane & 1) * (RQ / 2) + ((lane >> 1) & 1) * (RQ / 4))] = pacc[j];
  }
  main_sync();
  for (int r = threadIdx.x; r < sb; r += kT) {
    double t = red[r];
#pragma unroll
    for (int w = 1; w < 8; ++w) t += red[w * 8 * RQ + r];
    pp[r] = t;
  }
}

// Shared state of a column CTA's digit Gram; digits_begin / digits_end by all
// threads (tensor memory is held in between).
template <int RQ>
struct DigitShared {
  int emax[8 * RQ];
  float wt[8 * RQ];
  int nlist;
  uint32_t tmin[16];
  int64_t diag[RQ == 16 ? 128 : 1];
  uint64_t bars[5];
  uint32_t cmd[2];
  uint32_t tmem_holder;
};
// digits_begin, digits_end: the main warps and the MMA warp together (named
// barrier 9).
__device__ __forceinline__ void digit_sync() {
  asm volatile("bar.sync 9, %0;" ::"n"(kT + kMma) : "memory");
}
template <int RQ>
__device__ __forceinline__ void digits_begin(DigitGram<8 * RQ>& dg, DigitShared<RQ>& sh, void* smem) {
  dg.dig = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem) + 1023) &
                                            ~uintptr_t(1023));
  dg.bars = sh.bars;
  dg.emax = sh.emax;
  dg.wt = sh.wt;
  dg.nlist = &sh.nlist;
  dg.tmin = sh.tmin;
  dg.diag = sh.diag;
  dg.cmd = sh.cmd;
  if (threadIdx.x == 0) {
    for (int q = 0; q < 5; ++q) mbar_init(&sh.bars[q], q < 3 ? 1 : 8);
    fence_mbar_init();
  }
  if (threadIdx.x < 32) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sh.tmem_holder)),
                 "r"((uint32_t)DigitGram<8 * RQ>::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_proxy_async_smem();
  tc_fence_before();
  digit_sync();
  tc_fence_after();
  dg.tmem = sh.tmem_holder;
}
template <int RQ>
__device__ __forceinline__ void digits_end(const DigitGram<8 * RQ>& dg) {
  tc_fence_before();
  digit_sync();
  if (threadIdx.x < 32) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(dg.tmem),
                 "r"((uint32_t)DigitGram<8 * RQ>::kTmemCols)
                 : "memory");
  }
}

// Gram partial of the CTA's columns [c0, c1).  DIG: more than kSmallSB rows.
template <int RQ, bool DIG, bool PAIR = false>
__device__ __forceinline__ bool gram_columns(DigitGram<8 * RQ>& dg, const double* __restrict__ A,
                                             const long long* off, int sb, long long c0,
                                             long long c1, double* smem_d, double* __restrict__ part,
                                             int sbp, unsigned* err, bool ok) {
  if constexpr (!DIG) {
    gram_small(A, off, sb, c0, c1, smem_d, part, sbp);
  } else {
    // segments of equal length, whole 32-column stages
    const long long nst = (c1 - c0 + 31) / 32, nseg = (nst + kSeg / 32 - 1) / (kSeg / 32);
    for (long long g = 0; g < nseg && ok; ++g)
      ok = dg.template gram<PAIR>(A, off, sb, c0 + nst * g / nseg * 32,
                                  min(c1, c0 + nst * (g + 1) / nseg * 32), part, sbp, g > 0, err, ok);
  }
  return ok;
}

// The Gram pass alone (steps a2+a3): split-K partials over gridDim.x CTAs and
// the projection partials on v.  PAIR (more than 128 rows): blockIdx.y is a pair
// of groups of 64 rows, whose 128-row Gram the CTA forms and of which it stores
// the off-diagonal block, the diagonal block of a group being stored with the
// next group (the last one's with the first: both with the last pair made that
// one the last to end).  (ng - 1) ng / 2 tiles, of which a group pair is one;
// normal numbers 256 x 24001 0.33 ms, 512 x 24001 1.47 ms (1.80 and 6.42 ms as
// FP64 FMAs in 64 x 64 tiles); four fifths zeros 1.80 and 8.7 ms; elements of 24
// decades, every entry off the diagonal by FP64, 2.31 and 11.1 ms.
template <int RQ, bool DIG, bool PAIR>
__global__ void __launch_bounds__(kT + kMma, 1)
k_gram64(Persist64Args a, unsigned* __restrict__ err) {
  extern __shared__ double smem_d[];
  __shared__ long long soff[8 * RQ];
  __shared__ double ured[64 * RQ];
  __shared__ DigitShared<RQ> sh;
  const int P = (int)gridDim.x, c = blockIdx.x, sbp = a.sa.ldr;
  const long long nch = (a.K + 15) / 16;
  const long long c0 = nch * c / P * 16, c1 = min(a.K, nch * (c + 1) / P * 16);
  DigitGram<8 * RQ> dg;
  int sb = a.sb, ga = 0, gb = 1;  // rows, and the groups of a pair
  if constexpr (PAIR) {
    const int ng = (a.sb + 63) / 64;
    tri_decode((int)blockIdx.y, gb, ga);
    ++gb;
    sb = 64 + min(64, a.sb - 64 * gb);
    dg.lo = 64 * ga;
    dg.hi = 64 * (gb - 1);
    dg.own_lo = gb == ga + 1;
    dg.own_hi = ga == 0 && gb == ng - 1;
  }
  if constexpr (DIG) digits_begin<RQ>(dg, sh, smem_d);
  if (threadIdx.x >= kT) {
    if constexpr (DIG) {
      dg.mma_loop(err);
      digits_end<RQ>(dg);
    }
    return;
  }
  if constexpr (PAIR) {
    row_offsets(a.idx_all + 64 * ga, 64, a.N, a.lda, soff, err);
    row_offsets(a.idx_all + 64 * gb, sb - 64, a.N, a.lda, soff + 64, err);
  } else {
    row_offsets(a.idx_all, sb, a.N, a.lda, soff, err);
  }
  main_sync();
  gram_columns<RQ, DIG, PAIR>(dg, a.A, soff, sb, c0, c1, smem_d, a.part + (long long)c * sbp * sbp, sbp,
                         err, true);
  double* pp = a.ppart + (long long)c * sbp;
  if constexpr (PAIR) {
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      if (!(h == 0 ? dg.own_lo : dg.own_hi)) continue;
      update_project<RQ>(a, soff + 64 * h, soff, nullptr, h == 0 ? 64 : sb - 64, 0, c0, c1, ured,
                         pp + 64 * (h == 0 ? ga : gb));
      main_sync();  // (ured is free again)
    }
  } else {
    update_project<RQ>(a, soff, soff, nullptr, sb, 0, c0, c1, ured, pp);
  }
  if constexpr (DIG) {
    dg.stop();
    digits_end<RQ>(dg);
  }
}

// p[r] = the sum of the P partials of sb < kRowsSB rows, all threads.  An FP64
// addition holds a scheduler for 64 cycles whatever the lanes in use: for few
// rows a warp sums a row (lanes over the partials), for more the lanes take the
// rows and the warps share the partials (sm: 256 sums).
__device__ __forceinline__ void sum_rows(const Persist64Args& a, int P, int sbp, int sb, double* sm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (sb <= 8) {
    if (warp < sb) {
      double t = 0.0;
#pragma unroll 5
      for (int q = lane; q < P; q += 32) t += __ldcg(a.ppart + (long long)q * sbp + warp);
      for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) a.pvec[warp] = t;
    }
  } else {
    double t = 0.0;
    if (lane < sb) {
#pragma unroll 16
      for (int q = warp; q < P; q += 8) t += __ldcg(a.ppart + (long long)q * sbp + lane);
    }
    sm[threadIdx.x] = t;
    main_sync();
    if (warp == 0 && lane < sb) {
      for (int w = 1; w < 8; ++w) t += sm[lane + 32 * w];
      a.pvec[lane] = t;
    }
  }
  main_sync();
}

// Entries of the lower triangle a reducing CTA takes: as few as spread the E
// entries over the P CTAs (a power of two, 4 .. 32).
__device__ __forceinline__ int entries_a_role(int E, int P) {
  int epr = 4;
  while (epr < 32 && epr * P < E) epr *= 2;
  return epr;
}

// (DIG false, up to kSmallSB rows: a kernel of its own, whose registers the
// digits' loops have no part in: X 64 x 1024, s = 1 1.75 -> 1.69 ms, s = 4 0.64 ->
// 0.62 a solve)
template <int BMAX, int DEPTH, int RQ, bool DIG>
__global__ void __launch_bounds__(kT + kMma + kSide, 1)
k_persist64(Persist64Args a, unsigned* __restrict__ err) {
  extern __shared__ double smem_d[];
  const int tid = threadIdx.x;
  const int sb = a.sb, sbp = a.sa.ldr, npass = a.npass;
  const int b = a.sa.b, s = a.sa.s_cur;
  const int ninv = min(s, kMaxInv), P = (int)gridDim.x - 1 - ninv, c = blockIdx.x;
  const long long sq = (long long)sbp * sbp;
  const int E = sb * (sb + 1) / 2, epr = entries_a_role(E, P);
  const int nrole = (E + epr - 1) / epr, nred = min(P, nrole);  // roles and CTAs that reduce
  bool ok = true;

  if (c == P + ninv) {  // ----------------------------------------- chain CTA
    if (tid >= kT) return;
    for (int p = 0; p < npass; ++p) {
      const long long k = a.k0 + p;
      SolveArgs sa = a.sa;
      sa.idx = a.idx_all + k * sb;
      sa.delta = a.delta2[k & 1];
      const bool done = chain_la_body<BMAX, DEPTH>(
          a.Rs[k & 1], a.pvec, a.Ginv[k & 1], sa, err, smem_d, [&] {
            ok = main_wait(a.cnt + Cnt::R + (p & 1), (unsigned)(ninv * (p / 2 + 1)), err, ok);
            ok = sb >= kRowsSB ? main_wait(a.cnt + Cnt::Q, (unsigned)(min(P, sb) * (p + 1)), err, ok)
                               : main_wait(a.cnt + Cnt::P, (unsigned)(P * (p + 1)), err, ok);
            if (ok && sb < kRowsSB) sum_rows(a, P, sbp, sb, smem_d);
            return ok;
          });
      if (!done) return;
      main_count(a.cnt + Cnt::D);
    }
    return;
  }

  if (c >= P) {  // ------------------------------------------------ inverse CTA
    if (tid >= kT) return;
    __shared__ float2 colbuf[66];
    for (int p = 0; p < npass && ok; ++p) {
      ok = main_wait(a.cnt + Cnt::E + (p & 1), (unsigned)(nred * (p / 2 + 1)), err, ok);
      int done = 0;  // pivots: the blocks of this CTA share colbuf without a barrier between them
      for (int j = c - P; j < s; j += ninv, done += b) {  // (each block replaced by its inverse)
        float2* out = a.Ginv[(a.k0 + p) & 1] + (long long)j * b * b;
        float2 m[1] = {tid < b * b ? __ldcg(out + tid) : make_float2(0.f, 0.f)};
        if (BMAX > 8) cta_sweep_inverse<1, kT, 8>(m, b, colbuf, out, err, tid, done);
        else if (tid < 64) cta_sweep_inverse<1, 64, 8>(m, b, colbuf, out, err, tid, done);
      }
      main_count(a.cnt + Cnt::R + (p & 1));
    }
    return;
  }

  // --------------------------------------------------------------- column CTA
  __shared__ long long soff[2][8 * RQ];
  __shared__ double sdl[8 * RQ];  // zero past the rows
  __shared__ double ured[64 * RQ];
  if (tid >= kT + kMma) {
    // side warps: this CTA's share of each step's reduction, epr entries a role,
    // 96 / epr threads an entry
    __shared__ double red[kSide];
    const int st = tid - kT - kMma, sw = st >> 5, lane = st & 31;
    const float2 cG2 = split_f64(a.sa.cG), cI2 = split_f64(a.sa.cI);
    auto sync = [&]() { asm volatile("bar.sync %0, %1;" ::"n"(kBarSide), "n"(kSide) : "memory"); };
    auto count = [&](unsigned* p) {
      sync();
      if (st == 0) {
        __threadfence();
        atomicAdd(p, 1u);
      }
    };
    for (int p = 0; p < npass; ++p) {
      const long long k = a.k0 + p;
      if (c < nrole) {
        if (st == 0) wait_count(a.cnt + Cnt::G + (p & 1), (unsigned)(P * (p / 2 + 1)), err);
        sync();
        const double* part = a.part + (k & 1) * (long long)P * sq;
        float2* Gi = a.Ginv[k & 1];
        const int en = lane & (epr - 1), wsub = 32 / epr;  // threads of an entry in a warp
        for (int role = c; role < nrole; role += P) {
          const int e = role * epr + en;
          int i = 0, j = 0;
          double t = 0.0;
          if (e < E) {  // column-major over the lower triangle: lanes along i
            int ir, jr;
            tri_decode(e, ir, jr);
            i = sb - 1 - jr;
            j = sb - 1 - ir;
            const double* src = part + (long long)j * sbp + i;
#pragma unroll 16
            for (int q = sw * wsub + lane / epr; q < P; q += 3 * wsub) t += __ldcg(src + q * sq);
          }
          for (int o = 16; o >= epr; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
          red[st] = t;
          sync();
          if (st < epr && e < E) {
            float2 g = df_mul(cG2, split_f64((t + red[32 + st]) + red[64 + st]));
            const int bj = j / b, ii = i - bj * b, jj = j - bj * b;
            if (ii < b) {  // diagonal block bj: Gamma, for its inverse
              if (i == j) g = df_add(g, cI2);
              Gi[((long long)bj * b + ii) * b + jj] = g;
              Gi[((long long)bj * b + jj) * b + ii] = g;
            } else {
              a.Rs[k & 1][(long long)j * sbp + i] = g;
            }
          }
          sync();
        }
        count(a.cnt + Cnt::E + (p & 1));
      }
      if (sb >= kRowsSB && c < sb) {  // rows c, c + P, ... of p: lanes over the partials
        if (st == 0) wait_count(a.cnt + Cnt::P, (unsigned)(P * (p + 1)), err);
        sync();
        for (int r = c + P * sw; r < sb; r += 3 * P) {
          double t = 0.0;
#pragma unroll 5
          for (int q = lane; q < P; q += 32) t += __ldcg(a.ppart + (long long)q * sbp + r);
          for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
          if (lane == 0) a.pvec[r] = t;
        }
        count(a.cnt + Cnt::Q);
      }
    }
    return;
  }
  __shared__ DigitShared<RQ> sh;
  DigitGram<8 * RQ> dg;
  if constexpr (DIG) digits_begin<RQ>(dg, sh, smem_d);
  if (tid >= kT) {
    if constexpr (DIG) {
      dg.mma_loop(err);
      digits_end<RQ>(dg);
    }
    return;
  }
  const long long nch = (a.K + 15) / 16;  // (half stages: even shares)
  const long long c0 = nch * c / P * 16, c1 = min(a.K, nch * (c + 1) / P * 16);
  auto gram = [&](int p, const long long* off) {  // the partial of step k0 + p
    double* part = a.part + ((a.k0 + p) & 1) * (long long)P * sq;
    ok = gram_columns<RQ, DIG>(dg, a.A, off, sb, c0, c1, smem_d, part + c * sq, sbp, err, ok);
    main_count(a.cnt + Cnt::G + (p & 1));
  };

  row_offsets(a.idx_all + a.k0 * sb, sb, a.N, a.lda, soff[0], err);
  main_sync();
  gram(0, soff[0]);
  for (int p = 0; p < npass && ok; ++p) {
    const long long k = a.k0 + p;
    const int psb = p == 0 ? 0 : sb;  // (no update is pending where a run starts)
    if (p > 0) ok = main_wait(a.cnt + Cnt::D, (unsigned)p, err, ok);
    if (!ok) break;
    if (psb > 0) {
      for (int r = tid; r < 8 * RQ; r += kT)
        sdl[r] = r < psb ? __ldcg(a.delta2[(k - 1) & 1] + r) : 0.0;
      main_sync();
    }
    update_project<RQ>(a, soff[p & 1], soff[(p + 1) & 1], sdl, sb, psb, c0, c1, ured,
                       a.ppart + (long long)c * sbp);
    main_count(a.cnt + Cnt::P);
    if (p + 1 < npass) {
      row_offsets(a.idx_all + (k + 1) * sb, sb, a.N, a.lda, soff[(p + 1) & 1], err);
      main_sync();
      gram(p + 1, soff[(p + 1) & 1]);
    }
  }
  if constexpr (DIG) {
    dg.stop();
    digits_end<RQ>(dg);
  }
}

// Dynamic shared memory of a column CTA.  With digits more than half of an
// SM's: two launches never share an SM, so neither can hold the tensor memory
// that a CTA of the other, which its grid waits for, needs.
template <int RQ>
size_t column_smem(int sb) {
  if (sb <= kSmallSB) return (kSmallSB * 33 + 8 * (size_t)(kSmallSB * (kSmallSB + 1) / 2)) * 8;
  return std::max<size_t>(DigitGram<8 * RQ>::kSmem, 118 * 1024);
}

template <typename Kern>
int launch64(Kern kern, std::atomic<unsigned long long>& configured, const Persist64Args& a,
             dim3 grid, size_t smem, bool coop, unsigned* err, cudaStream_t st) {
  if (smem > (size_t)kSmemMax) return (int)cudaErrorInvalidConfiguration;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  const unsigned long long bit = dev < 64 ? (1ull << dev) : 0ull;  // a bit per device
  if (!bit || !(configured.load(std::memory_order_acquire) & bit)) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return (int)e;
    configured.fetch_or(bit, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(coop ? kT + kMma + kSide : kT + kMma);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;  // every CTA resident at once
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = coop ? 1 : 0;
  e = cudaLaunchKernelEx(&cfg, kern, a, err);
  return (int)(e != cudaSuccess ? e : cudaGetLastError());
}

template <int BMAX, int DEPTH, int RQ, bool DIG>
int launch_steps(const Persist64Args& a, int P, size_t chain_smem, unsigned* err, cudaStream_t st) {
  static std::atomic<unsigned long long> configured{0ull};
  return launch64(k_persist64<BMAX, DEPTH, RQ, DIG>, configured, a, P + 1 + std::min(a.sa.s_cur, kMaxInv),
                  std::max(chain_smem, column_smem<RQ>(a.sb)), true, err, st);
}

template <int RQ, bool DIG = true, bool PAIR = false>
int launch_gram(const Persist64Args& a, dim3 grid, unsigned* err, cudaStream_t st) {
  static std::atomic<unsigned long long> configured{0ull};
  return launch64(k_gram64<RQ, DIG, PAIR>, configured, a, grid, column_smem<RQ>(a.sb), false, err, st);
}

// pairs of groups of 64 rows (one: all rows in one CTA)
int gram64_pairs(int sb) {
  const int ng = (sb + 63) / 64;
  return sb <= 128 ? 1 : ng * (ng - 1) / 2;
}

}  // namespace

// One CTA per SM over the column splits and row pairs.
int gram64_splits(int sb, long long K, int num_sms) {
  return (int)std::min<long long>(std::max(1, num_sms / gram64_pairs(sb)), (K + 31) / 32);
}

int launch_gram64(const double* A, long long lda, long long N, long long K, const int* idx, int sb,
                  const double* v, int P, int sbp, double* part, double* ppart, unsigned* err,
                  cudaStream_t st) {
  Persist64Args a{};
  a.A = A;
  a.lda = lda;
  a.N = N;
  a.K = K;
  a.idx_all = idx;
  a.sb = sb;
  a.v = const_cast<double*>(v);  // read only: no update is pending
  a.part = part;
  a.ppart = ppart;
  a.sa.ldr = sbp;
  if (sb <= kSmallSB) return launch_gram<4, false>(a, dim3(P), err, st);
  if (sb <= 32) return launch_gram<4>(a, dim3(P), err, st);
  if (sb <= 64) return launch_gram<8>(a, dim3(P), err, st);
  if (sb <= 128) return launch_gram<16>(a, dim3(P), err, st);
  return launch_gram<16, true, true>(a, dim3(P, gram64_pairs(sb)), err, st);
}

int launch_persist64(const Persist64Args& a, int P, size_t chain_smem, unsigned* err,
                     cudaStream_t st) {
#define CA_P64(RQ, DIG)                                                       \
  return a.sa.b <= 8 ? launch_steps<8, 4, RQ, DIG>(a, P, chain_smem, err, st) \
                     : launch_steps<16, 3, RQ, DIG>(a, P, chain_smem, err, st);
  if (a.sb <= kSmallSB) CA_P64(4, false)
  if (a.sb <= 32) CA_P64(4, true)
  if (a.sb <= 64) CA_P64(8, true)
  if (a.sb <= 128) CA_P64(16, true)
#undef CA_P64
  return (int)cudaErrorInvalidValue;
}
