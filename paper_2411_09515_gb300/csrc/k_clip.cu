// Integration + sigma-clipping over staged pixel values.
//
// One warp owns one radial bin (a row of the integration matrix) of one
// frame: it reads the bin's values from the frame's staged copy (k_stage.cu:
// corrected pixels, Section 1.2, one slot per matrix entry, so a bin's
// values are one contiguous run), accumulates the weighted moments
// (Eqs. 8-13) and runs the clip loop of Eq. 19 (Section 2.4) by tail replay
// (described with the kernel below). The warps of a CTA take other frames
// of the same bin and wait for one another only when the CTA takes its next
// unit of work (a persistent launch draws units from a work-queue counter).
//
// Moments are accumulated about a shift K: with d = v - K, per set S
//   Omega = sum w, A1 = sum w d, OO = sum w^2, B1 = sum w^2 d, B2 = sum w^2 d^2,
//   mu = K + A1 / Omega,  VV = B2 - 2 (mu - K) B1 + (mu - K)^2 OO  (Eq. 11),
//   sigma = sqrt(VV / OO)  (Eq. 13),
// which is exact algebra; with K close to mu (or 0 where |mu| <= 2 sigma)
// the correction terms are small.
//
// Rejection is cumulative and symmetric about the current mean, so the set
// after t steps is every entry whose value lies in an interval [L_t, H_t]:
// no per-entry flag is kept. Row entries are grouped by coefficient class (a
// group shares one weight), so per-entry work is unweighted and the class
// weight is applied once per lane and class.
//
// After the last evaluation the kernel writes mu + k_pick sigma, the bin's
// sparsification threshold (Section 3); with a bitmap it also marks the
// bin's kept pixels (its centre entries above the threshold).
//
// Precision (SEP_PREC_*): per-lane FP32 sums (Kahan-compensated in KAHAN);
// the merge over the lanes and the finalisation in plain FP32 (PLAIN),
// error-free FP32 pairs ("double-word": KAHAN and DWORD, the default) or
// FP64 (FP64MERGE). FP64 runs at a small fraction of the FP32 rate on this
// GPU, so DWORD issues no FP64 instruction.
#include <cuda_runtime.h>
#include <float.h>
#include <stdint.h>

#include <algorithm>

#include "sep_device.cuh"
#include "sep_internal.h"
#include "sep_mlp.cuh"

namespace sep {
namespace {


enum { MODE_UNIT = 0, MODE_CLASS = 1, MODE_ENTRY = 2 };

template <bool KAHAN>
struct Acc {
  float s = 0.0f, c = 0.0f;   // value = s - c
  __device__ __forceinline__ void add(float x) {
    if (KAHAN) {
      const float y = __fsub_rn(x, c);
      const float t = __fadd_rn(s, y);
      c = __fsub_rn(__fsub_rn(t, s), y);
      s = t;
    } else {
      s = __fadd_rn(s, x);
    }
  }
  // += x * y: compensated product in KAHAN, one fused multiply-add otherwise
  __device__ __forceinline__ void add_prod(float x, float y) {
    if (KAHAN) add(__fmul_rn(x, y));
    else s = __fmaf_rn(x, y, s);
  }
  __device__ __forceinline__ float val() const { return KAHAN ? __fsub_rn(s, c) : s; }
};

// (s - c) += (so - co): error-free two-sum of the leading parts
__device__ __forceinline__ void pair_add(float& s, float& c, float so, float co) {
  const float t = __fadd_rn(s, so);
  const float bp = __fsub_rn(t, s);
  const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(so, bp));
  c = __fsub_rn(__fadd_rn(c, co), err);
  s = t;
}

// Shift of the next pass. With K = 0 the deviations d = v are exact, and
// the variance terms cancel by at most a factor 1 + mu^2 / sigma^2 <= 5 when
// |mu| <= 2 sigma; otherwise K = mu keeps the cancellation small and the
// rounding of d = v - K (relative 2^-24 of |d| ~ sigma) is far below the
// mean's own scale.
__device__ __forceinline__ float choose_shift(float mu, float sd) { return fabsf(mu) <= 2.0f * sd ? 0.0f : mu; }

// State of an item's clip loop (every lane of its warp holds the same
// copy, evaluated from bit-identical totals). The mean is kept as an
// unevaluated FP32 pair mu_hi + mu_lo (FP64MERGE keeps a double).
struct Bcast {
  double mu_d, sd_d;   // FP64MERGE
  float mu_hi, mu_lo, sd;
  float Ln, Hn, Kf;    // interval and shift of the next pass
  float L, H;          // interval of the current set
  float n_cur;         // entries (weight != 0) in the current set
  int steps, done;
  float sdP;           // Poisson deviation of the current set (error models 1, 2)
  double sdP_d;        // FP64MERGE
};

// Error-free sum: a + b = s + e exactly.
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bp = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bp)), __fsub_rn(b, bp));
}

// Smallest float >= hi + lo and largest float <= hi + lo for a normalised
// pair (hi = RN(hi + lo)).
// (next binary32 value up or down from its bit pattern; lo is NaN or 0, so
// hi stays, where hi is not finite)
__device__ __forceinline__ float round_up_pair(float hi, float lo) {
  const int b = __float_as_int(hi);
  const int up = hi == 0.0f ? 1 : b + (b < 0 ? -1 : 1);
  return lo > 0.0f ? __int_as_float(up) : hi;
}
__device__ __forceinline__ float round_dn_pair(float hi, float lo) { return -round_up_pair(-hi, -lo); }

// Mean and deviation of one set from its shifted sums (each lane of the
// item's warp, on the same totals):
//   mu = K + A1 / Omega,  VV = B2 - 2 (mu - K) B1 + (mu - K)^2 OO,  sd = sqrt(VV / OO)
// Sums arrive as FP32 pairs (value = hi + lo). The divisions act on a small
// correction and on a ratio, where FP32 is exact to ~1e-7 relative; the
// mean is kept as the exact pair K + corr. FP64MERGE does the same in FP64.
template <int PREC>
__device__ __forceinline__ void finalise(float Kf, const float (&hi)[6], const float (&lo)[6], Bcast& st) {
  // hi/lo layout: 0 Omega, 1 A1, 2 OO, 3 B1, 4 B2
  if (hi[0] == 0.0f) {
    st.mu_hi = st.mu_lo = st.sd = 0.0f;
    st.mu_d = st.sd_d = 0.0;
    return;
  }
  if (PREC == SEP_PREC_FP64MERGE) {
    const double Om = (double)hi[0] + lo[0], A1 = (double)hi[1] + lo[1], OO = (double)hi[2] + lo[2];
    const double B1 = (double)hi[3] + lo[3], B2 = (double)hi[4] + lo[4];
    const double mu = (double)Kf + (double)__fdiv_rn((float)A1, (float)Om);
    const double dl = mu - (double)Kf;
    const double VV = fma(dl * dl, OO, fma(-2.0 * dl, B1, B2));
    st.mu_d = mu;
    st.sd_d = VV > 0.0 ? (double)__fsqrt_rn(__fdiv_rn((float)VV, (float)OO)) : 0.0;
    st.mu_hi = (float)mu;
    st.mu_lo = (float)(mu - (double)st.mu_hi);
    st.sd = (float)st.sd_d;
    return;
  }
  const float Om = __fadd_rn(hi[0], lo[0]), OO = __fadd_rn(hi[2], lo[2]);
  const float corr = __fdiv_rn(__fadd_rn(hi[1], lo[1]), Om);
  if (PREC == SEP_PREC_PLAIN) {
    st.mu_hi = __fadd_rn(Kf, corr);
    st.mu_lo = 0.0f;
  } else {
    two_sum(Kf, corr, st.mu_hi, st.mu_lo);
  }
  // VV with the small correction terms in FP32 and the leading B2 as a pair
  float VV = __fsub_rn(hi[4], __fmul_rn(2.0f * corr, __fadd_rn(hi[3], lo[3])));
  VV = __fadd_rn(VV, __fmul_rn(__fmul_rn(corr, corr), OO));
  VV = __fadd_rn(VV, lo[4]);
  st.sd = VV > 0.0f ? __fsqrt_rn(__fdiv_rn(VV, OO)) : 0.0f;
}

// Next interval: keep |v - mu| <= k sd (Eq. 19). Except in PLAIN the float
// bounds are rounded outward-exact from the extended mean, so for any float
// v the test v >= L equals v >= mu - k sd up to the rounding of k sd.
template <int PREC>
__device__ __forceinline__ void clip_bounds(const Bcast& st, float k, float& L, float& H) {
  if (PREC == SEP_PREC_PLAIN) {
    const float ks = __fmul_rn(k, st.sd);
    L = fmaxf(L, __fsub_rn(st.mu_hi, ks));
    H = fminf(H, __fadd_rn(st.mu_hi, ks));
  } else if (PREC == SEP_PREC_FP64MERGE) {
    L = fmaxf(L, __double2float_ru(fma(-(double)k, st.sd_d, st.mu_d)));
    H = fminf(H, __double2float_rd(fma((double)k, st.sd_d, st.mu_d)));
  } else {
    const float ks = __fmul_rn(k, st.sd);
    float a, e;
    two_sum(st.mu_hi, -ks, a, e);
    e = __fadd_rn(e, st.mu_lo);
    float lh, ll;
    two_sum(a, e, lh, ll);
    L = fmaxf(L, round_up_pair(lh, ll));
    two_sum(st.mu_hi, ks, a, e);
    e = __fadd_rn(e, st.mu_lo);
    two_sum(a, e, lh, ll);
    H = fminf(H, round_dn_pair(lh, ll));
  }
}

// Threshold of sparsification, mu + k_pick sd, rounded down (v > thr is
// then the exact comparison for float v, up to the rounding of k sd).
template <int PREC>
__device__ __forceinline__ float pick_threshold(const Bcast& st, float k) {
  if (PREC == SEP_PREC_PLAIN) return __fadd_rn(st.mu_hi, __fmul_rn(k, st.sd));
  if (PREC == SEP_PREC_FP64MERGE) return __double2float_rd(fma((double)k, st.sd_d, st.mu_d));
  const float ks = __fmul_rn(k, st.sd);
  float a, e, th, tl;
  two_sum(st.mu_hi, ks, a, e);
  e = __fadd_rn(e, st.mu_lo);
  two_sum(a, e, th, tl);
  return round_dn_pair(th, tl);
}

template <int MODE>
struct Sums {
  // per pass, float sums and integer counts:
  //   MODE_UNIT:  (S1, S2) + count
  //   MODE_CLASS: (A1, B1, B2) + class counts packed 16 + 16 bits in two words
  //   MODE_ENTRY: (Omega, A1, OO, B1, B2) + count
  // (a row holds fewer than 2^16 entries: the host refuses longer rows; tail
  // slots keep an entry's index in 16 bits)
  static constexpr int NF = MODE == MODE_UNIT ? 2 : (MODE == MODE_CLASS ? 3 : 5);
  static constexpr int NI = MODE == MODE_CLASS ? 2 : 1;
};

// One step of the clip loop (every lane of the warp, on identical totals) after a pass measured the set
// S' = S ∩ [Ln, Hn] (count n_set, sums h/l about Kf). S' == S means nothing
// was discarded: the loop ends with the moments of S. Otherwise S' becomes
// the set, its moments are evaluated and the next interval is the
// intersection with [mu - k sd, mu + k sd] (Eq. 19, cumulative).
// (have_moments: st already holds the moments of S'.)
// Poisson deviation of a set (Eqs. 3-4, normalised as Eq. 13): each
// value's variance is the value plus the dark variance, weighted by the
// squared coefficients: sdP^2 = sum w^2 v / sum w^2 + dark = Kf + B1 / OO +
// dark from the pass's sums about Kf (0 when negative or the set is empty).
template <int PREC>
__device__ __forceinline__ void poisson_sd(float Kf, const float (&hi)[6], const float (&lo)[6], float dark,
                                           Bcast& st) {
  // hi/lo layout: 0 Omega, 1 A1, 2 OO, 3 B1, 4 B2
  if (hi[2] == 0.0f) {
    st.sdP = 0.0f;
    st.sdP_d = 0.0;
    return;
  }
  if (PREC == SEP_PREC_FP64MERGE) {
    const double OO = (double)hi[2] + lo[2], B1 = (double)hi[3] + lo[3];
    const double var = (double)Kf + B1 / OO + (double)dark;
    st.sdP_d = var > 0.0 ? sqrt(var) : 0.0;
    st.sdP = (float)st.sdP_d;
    return;
  }
  const float corr = __fdiv_rn(__fadd_rn(hi[3], lo[3]), __fadd_rn(hi[2], lo[2]));
  float s, e;
  two_sum(Kf, corr, s, e);
  const float var = __fadd_rn(s, __fadd_rn(e, dark));
  st.sdP = var > 0.0f ? __fsqrt_rn(var) : 0.0f;
  st.sdP_d = st.sdP;
}

// The reported (and, for the Poisson model, clipping) deviation becomes the
// Poisson one.
__device__ __forceinline__ void use_poisson(Bcast& st) {
  st.sd = st.sdP;
  st.sd_d = st.sdP_d;
}

// Chauvenet's cut-off for a set of n entries (Eq. 20): sqrt(2 ln(n / sqrt(2 pi))),
// n > 2 (FP32 library logarithm and square root).
__device__ __forceinline__ float chauvenet_k(float n) {
  return sqrtf(2.0f * logf(n * 0.3989422804014327f));
}

template <int PREC>
__device__ __forceinline__ void clip_step(Bcast& st, float n_set, const float (&h)[6], const float (&l)[6], float Kf,
                                          float Ln, float Hn, int n_iter, float k, bool have_moments = false,
                                          int cutoff = SEP_CUTOFF_FIXED, int model = SEP_ERROR_AZIMUTHAL,
                                          float dark = 0.0f) {
  if (st.steps >= 0 && n_set == st.n_cur) {
    if (model == SEP_ERROR_HYBRID) use_poisson(st);   // the final set's Poisson deviation
    st.done = 1;
    return;
  }
  st.n_cur = n_set;
  st.L = Ln;
  st.H = Hn;
  if (!have_moments) finalise<PREC>(Kf, h, l, st);
  if (model != SEP_ERROR_AZIMUTHAL) {
    poisson_sd<PREC>(Kf, h, l, dark, st);
    if (model == SEP_ERROR_POISSON) use_poisson(st);
  }
  st.steps += 1;
  // (Chauvenet: a set of two or fewer is not clipped, the loop ends here)
  if (st.steps >= n_iter || (cutoff == SEP_CUTOFF_CHAUVENET && n_set <= 2.0f)) {
    if (model == SEP_ERROR_HYBRID) use_poisson(st);
    st.done = 1;
    return;
  }
  if (cutoff == SEP_CUTOFF_CHAUVENET) k = chauvenet_k(n_set);
  float L2 = Ln, H2 = Hn;
  clip_bounds<PREC>(st, k, L2, H2);
  st.Ln = L2;
  st.Hn = H2;
  st.Kf = choose_shift(st.mu_hi, st.sd);
}

// A pass's totals as (count, Omega, A1, OO, B1, B2) pairs (every lane).
template <int MODE>
__device__ __forceinline__ void unpack_totals(const float* th, const float* tl, float& n_set, float (&h)[6],
                                              float (&l)[6]) {
#pragma unroll
  for (int v = 0; v < 6; ++v) h[v] = l[v] = 0.0f;
  if (MODE == MODE_CLASS) {
    // class counts are exact integers; their weighted sums are exact in FP32
    const uint32_t p01 = __float_as_uint(th[3]), p23 = __float_as_uint(th[4]);
    const float n0 = (float)(p01 & 0xffffu), n1 = (float)(p01 >> 16);
    const float n2 = (float)(p23 & 0xffffu), n3 = (float)(p23 >> 16);
    n_set = n0 + n1 + n2 + n3;
    h[0] = n0 + 0.75f * n1 + 0.5f * n2 + 0.25f * n3;
    h[2] = n0 + 0.5625f * n1 + 0.25f * n2 + 0.0625f * n3;
    h[1] = th[0]; l[1] = tl[0];
    h[3] = th[1]; l[3] = tl[1];
    h[4] = th[2]; l[4] = tl[2];
  } else if (MODE == MODE_UNIT) {
    n_set = (float)__float_as_uint(th[2]);
    h[0] = h[2] = n_set;
    h[1] = h[3] = th[0]; l[1] = l[3] = tl[0];
    h[4] = th[1]; l[4] = tl[1];
  } else {
    n_set = (float)__float_as_uint(th[5]);
#pragma unroll
    for (int v = 0; v < 5; ++v) { h[v] = th[v]; l[v] = tl[v]; }
  }
}

// ---------------------------------------------------------------------------
// Clip by tail replay, one warp per bin and frame (the plain path and the
// surrogate's record and inference variants).
//
// Every set of the clip loop is a value interval and the intervals are
// nested (Eq. 19 is cumulative). An interval C = [cLo, cHi] that lies inside
// every interval the loop has still to visit contributes the same entries,
// hence the same sums, to each remaining step; only the entries outside C
// (the tail) need to be tested again. Per bin and frame:
//   pass A  plain FP32 moments of the full set, used only to place C
//           kCoreMargin deviations inside the first clip interval;
//   pass B  one scan of the row: core entries are summed (in the call's
//           precision, about a shift K), every other valid entry is listed
//           in its lane's tail slots (value, entry index and class);
//   replay  the loop of Eq. 19 from the full set: the sums of a step are the
//           core sums plus a pass over the tail, finalised exactly as a full
//           pass would be (same set, sums in another order). When a new
//           interval no longer contains C, C is placed inside it and pass B
//           runs again; when a lane's tail slots overflow, the remaining
//           steps run as full passes.
// The kept-pixel marks come from the tail alone when the threshold lies at
// or above C (no core entry can exceed it), else from a scan of the row.
//
// A warp owns its item from the first load to the marks. The row is read
// from the staged frame (slot = entry, so a bin's values are one contiguous
// run) through a small ring (stream_row); only that and the tail live in
// shared memory, so many items fit an SM (15 for the longest rows of a
// Jungfrau 4M). The kernel is bound by its instructions (9,700 a bin and frame
// there: half of them the 5.5 replay steps, 40 % the scan of the row) at 61 %
// of the issue slots, which its 15 warps do not fill further: 48 Jungfrau-4M
// frames 925 -> 700 us, 4 frames 190 -> 150 us. Every total is a warp
// butterfly, which leaves bit-identical totals on all lanes (addition, and
// the error-free pair sum, are commutative), so every lane evaluates each
// clip step itself: no lane waits for another, and the warps of a CTA
// (other frames of the same bin) meet only between units of work.
constexpr float kCoreMargin = 1.0f;   // core margin inside the clip interval, in deviations
constexpr int kLoadsAhead = 4;        // 16-byte loads in flight per lane in a scan of the row
constexpr int kPairsAhead = 2;        // the same for a value and its weight
constexpr int kRing = 4;              // groups under way per lane in a walk of the row
constexpr int kMarkList = kRing * 256;  // kept entries a warp lists before their pixels are marked (16 bits each)
constexpr int kWarpsPerSM = 16;       // resident warps per SM the register budget is sized for

// One item's row: entry e's staged value at v4[e / 4] (padding slots NaN).
struct Row {
  const float4* v4;
};

// Scan of the 16-byte groups of [q0, q1) of a row by one lane of a
// warp: fn(v, q) for each of the lane's groups, kLoadsAhead loads issued
// before their use (groups past q1 are not loaded; fn is not called for
// them).
template <class F>
__device__ __forceinline__ void scan_row(const Row& row, int q0, int q1, int lane, F&& fn) {
  for (int q = q0 + lane; q < q1; q += 32 * kLoadsAhead) {
    float4 v[kLoadsAhead];
#pragma unroll
    for (int k = 0; k < kLoadsAhead; ++k)
      if (q + 32 * k < q1) v[k] = __ldg(row.v4 + q + 32 * k);
#pragma unroll
    for (int k = 0; k < kLoadsAhead; ++k)
      if (q + 32 * k < q1) fn(v[k], q + 32 * k);
  }
}

// The same for every step-th group with its entry weights: fn(v, w, q). The weights come
// through the read-only path like the values (every frame of the bin reads
// them, so all but the first reads hit the L2 or L1), two pairs at a time (three
// spill). Held in shared memory beside the tails they left room for 5 to 7
// warps on an SM; now 16 run: 1M pixels, 67 frames, norm, KAHAN 3046 -> 1560
// us; a ragged detector with area fractions, 131 frames, 604 -> 423 us (whole
// calls).
template <class F>
__device__ __forceinline__ void scan_weighted(const Row& row, const float* wts, int q0, int q1, int lane, F&& fn,
                                              int step = 1) {
  const float4* w4 = reinterpret_cast<const float4*>(wts);
  for (int q = q0 + lane * step; q < q1; q += 32 * step * kPairsAhead) {
    float4 v[kPairsAhead], w[kPairsAhead];
#pragma unroll
    for (int k = 0; k < kPairsAhead; ++k) {
      if (q + 32 * step * k < q1) {
        v[k] = __ldg(row.v4 + q + 32 * step * k);
        w[k] = __ldg(w4 + q + 32 * step * k);
      }
    }
#pragma unroll
    for (int k = 0; k < kPairsAhead; ++k)
      if (q + 32 * step * k < q1) fn(v[k], w[k], q + 32 * step * k);
  }
}

// Totals over the warp of NF per-lane sums (value s - c) as pairs
// hi + lo, identical on every lane: plain FP32 in PLAIN, doubles in
// FP64MERGE, error-free FP32 pairs otherwise.
template <int NF, int PREC>
__device__ __forceinline__ void warp_sum(const float (&s)[NF], const float (&c)[NF], float (&hi)[NF],
                                         float (&lo)[NF]) {
#pragma unroll
  for (int v = 0; v < NF; ++v) {
    if (PREC == SEP_PREC_PLAIN) {
      float x = s[v];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x = __fadd_rn(x, __shfl_xor_sync(0xffffffffu, x, o));
      hi[v] = x;
      lo[v] = 0.0f;
    } else if (PREC == SEP_PREC_FP64MERGE) {
      double t = (double)s[v] - (double)c[v];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      hi[v] = (float)t;
      lo[v] = (float)(t - (double)hi[v]);
    } else {
      float hs = s[v], hc = c[v];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float so = __shfl_xor_sync(0xffffffffu, hs, o);
        const float co = __shfl_xor_sync(0xffffffffu, hc, o);
        pair_add(hs, hc, so, co);
      }
      two_sum(hs, -hc, hi[v], lo[v]);
    }
  }
}

// Totals of a pass in the layout unpack_totals reads: NF float pairs, then
// the NI integer totals as raw bits.
template <int MODE, int PREC>
__device__ __forceinline__ void warp_totals(const float (&ss)[Sums<MODE>::NF], const float (&cc)[Sums<MODE>::NF],
                                            const uint32_t (&ci)[Sums<MODE>::NI], float& n_set, float (&h)[6],
                                            float (&l)[6]) {
  constexpr int NF = Sums<MODE>::NF, NI = Sums<MODE>::NI;
  float hi[NF], lo[NF];
  warp_sum<NF, PREC>(ss, cc, hi, lo);
  float th[NF + NI], tl[NF + NI];
#pragma unroll
  for (int v = 0; v < NF; ++v) {
    th[v] = hi[v];
    tl[v] = lo[v];
  }
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    th[NF + i] = __uint_as_float(__reduce_add_sync(0xffffffffu, ci[i]));
    tl[NF + i] = 0.0f;
  }
  unpack_totals<MODE>(th, tl, n_set, h, l);
}

// Class ends of a row, in groups of 4 entries (coefficient class c holds the
// groups [end(c - 1), end(c))).
struct ClassEnds {
  int e0, e1, e2, e3;
  __device__ __forceinline__ int end(int c) const { return c == 0 ? e0 : (c == 1 ? e1 : (c == 2 ? e2 : e3)); }
};

// Walk of a lane over its groups of every coefficient class in turn: from a
// class's first group on, the lane takes every 32nd of its every step-th
// groups, in blocks of kRing. quick(v, k, lo, c) gets group k of the block at
// lo of class c where all lanes have the whole block and room() holds (the
// same on all lanes), else fn(v, q, c) gets the lane's groups of the block
// one after another. close(c) follows the last group of each class, empty
// ones after the first group included.
//
// The groups come through the lane's own slots of a ring in shared memory, a
// block ahead of their use whatever class they belong to (16-byte cp.async
// copies; a lane reads only what it copied, so no barrier is needed): a
// warp's loads stay in flight through the whole row. With register loads, a
// block at a time and each class by itself, a warp waited for memory at every
// block (3.2 of the 7.3 cycles an instruction).
template <int NCLS, class R, class Q, class F, class C>
__device__ __forceinline__ void stream_row(const Row& row, const ClassEnds& ge, int lane, int step, uint32_t ring,
                                           R&& room, Q&& quick, F&& fn, C&& close) {
  const int hop = 32 * step, mine = lane * step;
  auto settle = [&](int& c, int& lo, int& hi) {   // to the next class with groups left
    if (NCLS > 1) {
      while (lo >= hi && c + 1 < NCLS) {
        lo = hi;
        ++c;
        hi = ge.end(c);
      }
    }
  };
  int c = 0, lo = 0, hi = ge.e0;
  settle(c, lo, hi);   // (leading empty classes have nothing to close: all sums are 0)
  // copies of the block of kRing groups from `p` on, of which the lane has
  // `left` groups of 32 step each to the class's end
  auto issue = [&](const float4* p, int left) {
#pragma unroll
    for (int k = 0; k < kRing; ++k)
      if (hop * k < left)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ring + 512u * k), "l"(p + hop * k) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto take = [&](int k) {   // group k of the block that has arrived
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(ring + 512u * k) : "memory");
    return v;
  };
  issue(row.v4 + lo + mine, hi - lo - mine);
#pragma unroll 1
  while (lo < hi) {
    int nc = c, nlo = lo + hop * kRing, nhi = hi;
    settle(nc, nlo, nhi);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (lo + hop * kRing <= hi && room()) {
      float4 v[kRing];
#pragma unroll
      for (int k = 0; k < kRing; ++k) v[k] = take(k);
      issue(row.v4 + nlo + mine, nhi - nlo - mine);   // under way while this block is used
#pragma unroll
      for (int k = 0; k < kRing; ++k) quick(v[k], k, lo, c);
    } else {
#pragma unroll 1
      for (int k = 0; lo + hop * k < hi && k < kRing; ++k)
        if (lo + hop * k + mine < hi) fn(take(k), lo + hop * k + mine, c);
      issue(row.v4 + nlo + mine, nhi - nlo - mine);
    }
    for (const int stop = nlo < nhi ? nc : NCLS; c < stop; ++c) close(c);
    c = nc;
    lo = nlo;
    hi = nhi;
  }
}

// A coefficient class's weight (1, 3/4, 1/2, 1/4).
__device__ __forceinline__ float class_weight(int c) { return 1.0f - 0.25f * (float)c; }

// Pass A (one lane's share): plain FP32 sums about 0 of the finite entries
// of every `step`-th group of 4 (a sample of a long row: they only place
// the core), in the layout unpack_totals reads (per-lane values).
template <int MODE>
__device__ __forceinline__ void lane_full_sums(const Row& row, const float* wts, const ClassEnds& ge,
                                               int lane, int step, uint32_t ring, float (&ss)[Sums<MODE>::NF],
                                               uint32_t (&ci)[Sums<MODE>::NI]) {
  constexpr int NF = Sums<MODE>::NF, NI = Sums<MODE>::NI;
#pragma unroll
  for (int v = 0; v < NF; ++v) ss[v] = 0.0f;
#pragma unroll
  for (int i = 0; i < NI; ++i) ci[i] = 0u;
  if (MODE == MODE_CLASS || MODE == MODE_UNIT) {
    uint32_t cnt = 0;
    float s1 = 0.0f, s2 = 0.0f;
    auto add = [&](const float4& v4) {
      const float xs[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        // finite entries (padding slots hold NaN)
        asm("{\n\t.reg .pred p;\n\t.reg .f32 m;\n\t"
            "abs.f32 m, %3;\n\t"
            "setp.le.f32 p, m, 0f7f7fffff;\n\t"
            "@p add.u32 %0, %0, 1;\n\t"
            "@p add.rn.f32 %1, %1, %3;\n\t"
            "@p fma.rn.f32 %2, %3, %3, %2;\n\t}"
            : "+r"(cnt), "+f"(s1), "+f"(s2) : "f"(xs[j]));
      }
    };
    stream_row<MODE == MODE_CLASS ? 4 : 1>(
        row, ge, lane, step, ring, [] { return true; }, [&](const float4& v4, int, int, int) { add(v4); },
        [&](const float4& v4, int, int) { add(v4);
    }, [&](int cls) {
      if (MODE == MODE_CLASS) {
        const float w = class_weight(cls), w2 = w * w;
        const uint32_t pk = cnt << (16 * (cls & 1));
        if (cls < 2) ci[0] += pk;
        else ci[NI - 1] += pk;
        ss[0] = fmaf(w, s1, ss[0]);
        ss[1] = fmaf(w2, s1, ss[1]);
        ss[2] = fmaf(w2, s2, ss[2]);
        cnt = 0;
        s1 = s2 = 0.0f;
      } else {
        ci[0] = cnt;
        ss[0] = s1;
        ss[1] = s2;
      }
    });
  } else {
    uint32_t cnt = 0;
    float om = 0.0f, a1 = 0.0f, oo = 0.0f, b1 = 0.0f, b2 = 0.0f;
    scan_weighted(row, wts, 0, ge.e3, lane, [&](const float4& v4, const float4& w4, int) {
      const float xs[4] = {v4.x, v4.y, v4.z, v4.w}, ws[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float w = ws[j];
        if (w != 0.0f && fabsf(xs[j]) <= FLT_MAX) {
          const float w2 = __fmul_rn(w, w), w2d = __fmul_rn(w2, xs[j]);
          ++cnt;
          om = __fadd_rn(om, w);
          a1 = __fmaf_rn(w, xs[j], a1);
          oo = __fadd_rn(oo, w2);
          b1 = __fadd_rn(b1, w2d);
          b2 = __fmaf_rn(w2d, xs[j], b2);
        }
      }
    }, step);
    ci[0] = cnt;
    ss[0] = om; ss[1] = a1; ss[2] = oo; ss[3] = b1; ss[4] = b2;
  }
}

// Pass B (one lane's share): sums about Kf of the entries inside
// [cLo, cHi] (the layout unpack_totals reads); every other valid entry goes to the
// lane's tail: slot k at tl[32 k] = (value bits, entry index | the upper half
// of its class weight's bits, or with entry weights the weight's bits), m
// slots in all. Returns false when a group of
// 4 entries found fewer than 4 of the tcap slots left (the sums are then
// incomplete).
template <int MODE, bool KAHAN>
__device__ __forceinline__ bool lane_core_sums(const Row& row, const float* wts, const ClassEnds& ge, int lane,
                                               float cLo, float cHi, float Kf, uint2* tl, int tcap, uint32_t ring, int& m,
                                               float (&ss)[Sums<MODE>::NF], float (&cc)[Sums<MODE>::NF],
                                               uint32_t (&ci)[Sums<MODE>::NI]) {
  constexpr int NF = Sums<MODE>::NF, NI = Sums<MODE>::NI;
#pragma unroll
  for (int v = 0; v < NF; ++v) ss[v] = cc[v] = 0.0f;
#pragma unroll
  for (int i = 0; i < NI; ++i) ci[i] = 0u;
  m = 0;
  bool fit = true;
  if (MODE == MODE_CLASS || MODE == MODE_UNIT) {
    float cnt = 0.0f;   // (exact: a row holds fewer than 2^16 entries)
    Acc<KAHAN> a1, a2;
    uint32_t at = (uint32_t)__cvta_generic_to_shared(tl);      // the lane's next tail slot
    const uint32_t at0 = at, most = at + 256u * (uint32_t)(tcap - 4);   // 4 slots left
    // one entry: into the sums, or into the tail, or (NaN) neither
    auto put = [&](float x, uint32_t tag) {
      if (KAHAN) {
        if (x >= cLo && x <= cHi) {
          const float d = __fsub_rn(x, Kf);
          cnt += 1.0f;
          a1.add(d);
          a2.add_prod(d, d);
        } else if (x == x) {
          asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(at), "r"(__float_as_uint(x)), "r"(tag) : "memory");
          at += 256u;
        }
      } else {
        // without a branch: most groups of a warp hold both kinds
        asm volatile(
            "{\n\t.reg .pred core, out;\n\t.reg .f32 d;\n\t"
            "setp.ge.f32 core, %4, %6;\n\t"
            "setp.le.and.f32 core, %4, %7, core;\n\t"
            "setp.num.and.f32 out, %4, %4, !core;\n\t"
            "sub.rn.f32 d, %4, %8;\n\t"
            "@core add.rn.f32 %0, %0, d;\n\t"
            "@core fma.rn.f32 %1, d, d, %1;\n\t"
            "@core add.rn.f32 %2, %2, 0f3f800000;\n\t"
            "@out st.shared.v2.b32 [%3], {%4, %5};\n\t"
            "@out add.u32 %3, %3, 256;\n\t}"
            : "+f"(a1.s), "+f"(a2.s), "+f"(cnt), "+r"(at)
            : "f"(x), "r"(tag), "f"(cLo), "f"(cHi), "f"(Kf)
            : "memory");
      }
    };
    auto tag_of = [&](int q, int cls) {
      return (uint32_t)(4 * q) | (MODE == MODE_CLASS ? __float_as_uint(class_weight(cls)) : 0u);
    };
    stream_row<MODE == MODE_CLASS ? 4 : 1>(
        row, ge, lane, 1, ring,
        // no lane can run out of slots within a block
        [&] { return !__any_sync(0xffffffffu, (int32_t)(at + 256u * 4 * (kRing - 1) - most) > 0); },
        [&](const float4& v4, int k, int lo, int cls) {
          const uint32_t tag = tag_of(lo + lane, cls) + 128u * k;
          put(v4.x, tag);
          put(v4.y, tag + 1);
          put(v4.z, tag + 2);
          put(v4.w, tag + 3);
        },
        [&](const float4& v4, int q, int cls) {
          if ((int32_t)(at - most) > 0) {
            fit = false;
          } else {
            const uint32_t tag = tag_of(q, cls);
            put(v4.x, tag);
            put(v4.y, tag + 1);
            put(v4.z, tag + 2);
            put(v4.w, tag + 3);
          }
    }, [&](int cls) {
      const float s1 = a1.val(), s2 = a2.val();
      if (MODE == MODE_CLASS) {
        const float w = class_weight(cls), w2 = w * w;
        const uint32_t pk = (uint32_t)cnt << (16 * (cls & 1));
        if (cls < 2) ci[0] += pk;
        else ci[NI - 1] += pk;
        if (KAHAN) {
          Acc<true> t0, t1, t2;
          t0.s = ss[0]; t0.c = cc[0]; t0.add(__fmul_rn(w, s1)); ss[0] = t0.s; cc[0] = t0.c;
          t1.s = ss[1]; t1.c = cc[1]; t1.add(__fmul_rn(w2, s1)); ss[1] = t1.s; cc[1] = t1.c;
          t2.s = ss[2]; t2.c = cc[2]; t2.add(__fmul_rn(w2, s2)); ss[2] = t2.s; cc[2] = t2.c;
        } else {
          ss[0] = fmaf(w, s1, ss[0]);
          ss[1] = fmaf(w2, s1, ss[1]);
          ss[2] = fmaf(w2, s2, ss[2]);
        }
        cnt = 0.0f;
        a1 = Acc<KAHAN>();
        a2 = Acc<KAHAN>();
      } else {
        ci[0] = (uint32_t)cnt;
        ss[0] = a1.s; cc[0] = a1.c; ss[1] = a2.s; cc[1] = a2.c;
      }
    });
    m = (int)((at - at0) >> 8);
    if (!fit) return false;
  } else {
    uint32_t cnt = 0;
    Acc<KAHAN> om, a1, oo, b1, b2;
    scan_weighted(row, wts, 0, ge.e3, lane, [&](const float4& v4, const float4& w4, int) {
      if (m + 4 > tcap) fit = false;
      if (!fit) return;
      const float xs[4] = {v4.x, v4.y, v4.z, v4.w}, ws[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float w = ws[j];
        if (w == 0.0f) continue;
        if (xs[j] >= cLo && xs[j] <= cHi) {
          const float d = __fsub_rn(xs[j], Kf);
          const float w2 = __fmul_rn(w, w);
          const float w2d = __fmul_rn(w2, d);
          ++cnt;
          om.add(w);
          a1.add(__fmul_rn(w, d));
          oo.add(w2);
          b1.add(w2d);
          b2.add_prod(w2d, d);
        } else if (xs[j] == xs[j]) {
          tl[32 * m] = make_uint2(__float_as_uint(xs[j]), __float_as_uint(w));
          ++m;
        }
      }
    });
    if (!fit) return false;
    ci[0] = cnt;
    ss[0] = om.s; cc[0] = om.c; ss[1] = a1.s; cc[1] = a1.c; ss[2] = oo.s; cc[2] = oo.c;
    ss[3] = b1.s; cc[3] = b1.c; ss[4] = b2.s; cc[4] = b2.c;
  }
  return true;
}

// One lane's share of a full pass over [Ln, Hn] about Kf (the layout
// unpack_totals reads), read from the staged row.
template <int MODE, bool KAHAN>
__device__ __noinline__ void lane_range_sums(const Row& row, const float* wts, const ClassEnds& ge,
                                                int lane, float Ln, float Hn, float Kf, uint32_t ring,
                                                float (&ss)[Sums<MODE>::NF], float (&cc)[Sums<MODE>::NF],
                                                uint32_t (&ci)[Sums<MODE>::NI]) {
  constexpr int NF = Sums<MODE>::NF, NI = Sums<MODE>::NI;
#pragma unroll
  for (int v = 0; v < NF; ++v) ss[v] = cc[v] = 0.0f;
#pragma unroll
  for (int i = 0; i < NI; ++i) ci[i] = 0u;
  if (MODE == MODE_CLASS || MODE == MODE_UNIT) {
    uint32_t cnt = 0;
    Acc<KAHAN> a1, a2;
    auto add = [&](const float4& v4) {
      const float xs[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (KAHAN) {
          if (xs[j] >= Ln && xs[j] <= Hn) {
            const float d = __fsub_rn(xs[j], Kf);
            ++cnt;
            a1.add(d);
            a2.add_prod(d, d);
          }
        } else {
          asm("{\n\t.reg .pred p;\n\t.reg .f32 d;\n\t"
              "setp.ge.f32 p, %3, %4;\n\t"
              "setp.le.and.f32 p, %3, %5, p;\n\t"
              "sub.rn.f32 d, %3, %6;\n\t"
              "@p add.u32 %0, %0, 1;\n\t"
              "@p add.rn.f32 %1, %1, d;\n\t"
              "@p fma.rn.f32 %2, d, d, %2;\n\t}"
              : "+r"(cnt), "+f"(a1.s), "+f"(a2.s)
              : "f"(xs[j]), "f"(Ln), "f"(Hn), "f"(Kf));
        }
      }
    };
    stream_row<MODE == MODE_CLASS ? 4 : 1>(
        row, ge, lane, 1, ring, [] { return true; }, [&](const float4& v4, int, int, int) { add(v4); },
        [&](const float4& v4, int, int) { add(v4);
    }, [&](int cls) {
      const float s1 = a1.val(), s2 = a2.val();
      if (MODE == MODE_CLASS) {
        const float w = class_weight(cls), w2 = w * w;
        const uint32_t pk = cnt << (16 * (cls & 1));
        if (cls < 2) ci[0] += pk;
        else ci[NI - 1] += pk;
        if (KAHAN) {
          Acc<true> t0, t1, t2;
          t0.s = ss[0]; t0.c = cc[0]; t0.add(__fmul_rn(w, s1)); ss[0] = t0.s; cc[0] = t0.c;
          t1.s = ss[1]; t1.c = cc[1]; t1.add(__fmul_rn(w2, s1)); ss[1] = t1.s; cc[1] = t1.c;
          t2.s = ss[2]; t2.c = cc[2]; t2.add(__fmul_rn(w2, s2)); ss[2] = t2.s; cc[2] = t2.c;
        } else {
          ss[0] = fmaf(w, s1, ss[0]);
          ss[1] = fmaf(w2, s1, ss[1]);
          ss[2] = fmaf(w2, s2, ss[2]);
        }
        cnt = 0;
        a1 = Acc<KAHAN>();
        a2 = Acc<KAHAN>();
      } else {
        ci[0] = cnt;
        ss[0] = a1.s; cc[0] = a1.c; ss[1] = a2.s; cc[1] = a2.c;
      }
    });
  } else {
    uint32_t cnt = 0;
    Acc<KAHAN> om, a1, oo, b1, b2;
    scan_weighted(row, wts, 0, ge.e3, lane, [&](const float4& v4, const float4& w4, int) {
      const float xs[4] = {v4.x, v4.y, v4.z, v4.w}, ws[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float w = ws[j];
        if (w != 0.0f && xs[j] >= Ln && xs[j] <= Hn) {
          const float d = __fsub_rn(xs[j], Kf);
          const float w2 = __fmul_rn(w, w);
          const float w2d = __fmul_rn(w2, d);
          ++cnt;
          om.add(w);
          a1.add(__fmul_rn(w, d));
          oo.add(w2);
          b1.add(w2d);
          b2.add_prod(w2d, d);
        }
      }
    });
    ci[0] = cnt;
    ss[0] = om.s; cc[0] = om.c; ss[1] = a1.s; cc[1] = a1.c; ss[2] = oo.s; cc[2] = oo.c;
    ss[3] = b1.s; cc[3] = b1.c; ss[4] = b2.s; cc[4] = b2.c;
  }
}

// One lane's tail entries inside [Ln, Hn]: (Omega, A1, OO, B1, B2) about Kf
// and their count (m: the lane's slots). Four entries at a time, so their
// reads are under way together.
template <int MODE, bool KAHAN>
__device__ __forceinline__ void lane_tail_sums(const uint2* tl, int m, float Ln, float Hn,
                                               float Kf, float (&ss)[5], float (&cc)[5], uint32_t& cnt) {
  Acc<KAHAN> acc[5];
  cnt = 0;
#pragma unroll 1
  for (int k0 = 0; k0 < m; k0 += 4) {
    uint2 t[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      t[u] = make_uint2(0x7fc00000u, 0u);   // NaN: in no interval
      if (k0 + u < m) t[u] = tl[32 * (k0 + u)];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float v = __uint_as_float(t[u].x);
      const float w = MODE == MODE_CLASS ? __uint_as_float(t[u].y & 0xffff0000u)
                                         : (MODE == MODE_UNIT ? 1.0f : __uint_as_float(t[u].y));
      if (KAHAN) {
        if (v >= Ln && v <= Hn) {
          const float d = __fsub_rn(v, Kf);
          const float w2 = __fmul_rn(w, w);
          const float w2d = __fmul_rn(w2, d);
          ++cnt;
          acc[0].add(w);
          acc[1].add(__fmul_rn(w, d));
          acc[2].add(w2);
          acc[3].add(w2d);
          acc[4].add_prod(w2d, d);
        }
      } else if (MODE == MODE_UNIT) {   // (unit weights: Omega = OO = count, B1 = A1)
        asm("{\n\t.reg .pred p;\n\t.reg .f32 d;\n\t"
            "setp.ge.f32 p, %3, %4;\n\t"
            "setp.le.and.f32 p, %3, %5, p;\n\t"
            "sub.rn.f32 d, %3, %6;\n\t"
            "@p add.u32 %0, %0, 1;\n\t"
            "@p add.rn.f32 %1, %1, d;\n\t"
            "@p fma.rn.f32 %2, d, d, %2;\n\t}"
            : "+r"(cnt), "+f"(acc[1].s), "+f"(acc[4].s)
            : "f"(v), "f"(Ln), "f"(Hn), "f"(Kf));
      } else {
        asm("{\n\t.reg .pred p;\n\t.reg .f32 d, w2, wd, w2d;\n\t"
            "setp.ge.f32 p, %6, %8;\n\t"
            "setp.le.and.f32 p, %6, %9, p;\n\t"
            "sub.rn.f32 d, %6, %10;\n\t"
            "mul.rn.f32 w2, %7, %7;\n\t"
            "mul.rn.f32 wd, %7, d;\n\t"
            "mul.rn.f32 w2d, w2, d;\n\t"
            "@p add.u32 %0, %0, 1;\n\t"
            "@p add.rn.f32 %1, %1, %7;\n\t"
            "@p add.rn.f32 %2, %2, wd;\n\t"
            "@p add.rn.f32 %3, %3, w2;\n\t"
            "@p add.rn.f32 %4, %4, w2d;\n\t"
            "@p fma.rn.f32 %5, w2d, d, %5;\n\t}"
            : "+r"(cnt), "+f"(acc[0].s), "+f"(acc[1].s), "+f"(acc[2].s), "+f"(acc[3].s), "+f"(acc[4].s)
            : "f"(v), "f"(w), "f"(Ln), "f"(Hn), "f"(Kf));
      }
    }
  }
  if (!KAHAN && MODE == MODE_UNIT) {
    acc[0].s = acc[2].s = (float)cnt;
    acc[3].s = acc[1].s;
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    ss[v] = acc[v].s;
    cc[v] = acc[v].c;
  }
}

// Totals over the warp of the five tail sums (hi + lo, identical on every
// lane). Sums of class weights and of their squares are multiples of 1/16
// that binary32 holds exactly whatever their order: they travel as integers
// (at most 177 entries a lane: 4 Omega below 2^15, 16 OO below 2^17), and
// with unit weights they are the count.
template <int MODE, int PREC>
__device__ __forceinline__ void tail_totals(const float (&ts)[5], const float (&tc)[5], uint32_t count, float (&th)[5],
                                            float (&tl)[5]) {
  if (MODE == MODE_ENTRY) {
    warp_sum<5, PREC>(ts, tc, th, tl);
    return;
  }
  if (MODE == MODE_UNIT) {
    th[0] = th[2] = (float)count;
  } else {
    const uint32_t mine = (uint32_t)(4.0f * ts[0]) + ((uint32_t)(16.0f * ts[2]) << 15);
    const uint32_t all = __reduce_add_sync(0xffffffffu, mine);
    th[0] = 0.25f * (float)(all & 0x7fffu);
    th[2] = 0.0625f * (float)(all >> 15);
  }
  tl[0] = tl[2] = 0.0f;
  constexpr int N = MODE == MODE_UNIT ? 2 : 3;
  float s[N], c[N], h[N], l[N];
  s[0] = ts[1]; c[0] = tc[1];
  s[1] = ts[4]; c[1] = tc[4];
  if (N > 2) { s[N - 1] = ts[3]; c[N - 1] = tc[3]; }
  warp_sum<N, PREC>(s, c, h, l);
  th[1] = h[0]; tl[1] = l[0];
  th[4] = h[1]; tl[4] = l[1];
  th[3] = h[N > 2 ? N - 1 : 0]; tl[3] = l[N > 2 ? N - 1 : 0];
}

// (h, l) += (a, b) for pairs, in the arithmetic of the precision mode.
template <int PREC>
__device__ __forceinline__ void add_pair(float& h, float& l, float a, float b) {
  if (PREC == SEP_PREC_PLAIN) {
    h = __fadd_rn(h, a);
  } else if (PREC == SEP_PREC_FP64MERGE) {
    const double t = ((double)h + (double)l) + ((double)a + (double)b);
    h = (float)t;
    l = (float)(t - (double)h);
  } else {
    float s, e;
    two_sum(h, a, s, e);
    e = __fadd_rn(e, __fadd_rn(l, b));
    two_sum(s, e, h, l);
  }
}

// ---- surrogate (no counterpart in the paper): features and inference ----
//
// Features of an item: 0 log(n) / 8 with n the valid entries of pass A's
// sample (every step-th group of 4 entries) times step, 1 Omega / n over
// that sample, 2 clamp(m1 / s1, -20, 20) / 4 with m1, s1 the sample's mean
// and Eq. 13 deviation; then, over a stratified subsample of at most 128 of
// the row's valid entries (sketch_element), 3 the share with z = (v - m1) /
// s1 >= 4 and 4 .. 19 the order statistics of z at ranks floor((j + 1/2)
// n' / 16) (n' the subsample's size; z clamped to [-4, 12]). The subsample
// is one 16-byte load per lane and four values a lane, sorted across the
// warp by a bitonic network.
constexpr float kSurrMargin = 0.5f;   // core margin inside the predicted final interval, in deviations

// Entry of the row behind sketch element s (0 .. 127) of a row whose first
// G groups of 4 hold its weighted entries: every entry when the row has at
// most 128 of them, else one entry of group floor(s G / 128) (-1: none).
__device__ __forceinline__ int sketch_element(int s, int G) {
  if (4 * G <= 128) return s < 4 * G ? s : -1;
  return 4 * (int)(((long long)s * G) >> 7) + (s & 3);
}

template <int MODE>
__device__ __forceinline__ void sample_features(const Row& row, const float* wts, const ClassEnds& ge, int lane,
                                                int step, float n_s, float om_s, float m1, float s1,
                                                float (&feat)[kIn]) {
  const int G = ge.e3;
  // element s = 32 r + lane of the sketch in x[r] (+inf where none)
  float x[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int e = sketch_element(32 * r + lane, G);
    float v = INFINITY;
    if (e >= 0) {
      const float4 q = __ldg(row.v4 + (e >> 2));
      const float c = (e & 3) == 0 ? q.x : ((e & 3) == 1 ? q.y : ((e & 3) == 2 ? q.z : q.w));
      const bool ok = fabsf(c) <= FLT_MAX && (MODE != MODE_ENTRY || __ldg(wts + e) != 0.0f);
      v = ok ? c : INFINITY;
    }
    x[r] = v;
  }
  // ascending bitonic sort of the 128 elements (index 32 r + lane)
#pragma unroll
  for (int k = 2; k <= 128; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      float y[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) y[r] = j >= 32 ? x[r ^ (j >> 5)] : __shfl_xor_sync(0xffffffffu, x[r], j);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int e = 32 * r + lane;
        const bool up = (e & k) == 0, low = (e & j) == 0;
        x[r] = (low == up) ? fminf(x[r], y[r]) : fmaxf(x[r], y[r]);
      }
    }
  }
  int nv = 0, hi4 = 0;
  const float z4 = fmaf(4.0f, s1, m1);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    nv += __popc(__ballot_sync(0xffffffffu, x[r] <= FLT_MAX));
    hi4 += __popc(__ballot_sync(0xffffffffu, x[r] <= FLT_MAX && x[r] >= z4));
  }
  const float inv = s1 > 0.0f ? 1.0f / s1 : 0.0f;
  const float n_est = n_s * (float)step;
  feat[0] = n_est > 0.0f ? logf(n_est) * 0.125f : 0.0f;
  feat[1] = n_s > 0.0f ? om_s / n_s : 0.0f;
  feat[2] = s1 > 0.0f ? fminf(fmaxf(m1 / s1, -20.0f), 20.0f) * 0.25f : 0.0f;
  feat[3] = nv > 0 ? (float)hi4 / (float)nv : 0.0f;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const int p = ((2 * j + 1) * nv) >> 5;   // floor((j + 1/2) nv / 16)
    const int r = p >> 5;
    const float mine = r == 0 ? x[0] : (r == 1 ? x[1] : (r == 2 ? x[2] : x[3]));
    const float q = __shfl_sync(0xffffffffu, mine, p & 31);
    feat[4 + j] = nv > 0 ? fminf(fmaxf(__fmul_rn(__fsub_rn(q, m1), inv), -4.0f), 12.0f) : 0.0f;
  }
}

// The network on one warp (weights BF16 with W1 and W2 input-major, FP32
// arithmetic; W and nm in shared memory): lane l computes hidden units l and l + 32 of each layer, so
// the warp reads consecutive weights; every lane returns the de-normalised
// outputs (mean offset, log-deviation ratio).
__device__ __forceinline__ void warp_mlp(const __nv_bfloat16* W, const float* nm, const float (&feat)[kIn], int lane,
                                         float& u0, float& u1) {
  float a1[2] = {__bfloat162float(W[kB1 + lane]), __bfloat162float(W[kB1 + lane + 32])};
#pragma unroll
  for (int k = 0; k < kIn; ++k) {
    const float xk = (feat[k] - nm[k]) / nm[kIn + k];
    a1[0] = fmaf(__bfloat162float(W[kW1 + k * kH + lane]), xk, a1[0]);
    a1[1] = fmaf(__bfloat162float(W[kW1 + k * kH + lane + 32]), xk, a1[1]);
  }
  const float h1[2] = {gelu_f(a1[0]), gelu_f(a1[1])};
  // layer 2: every input unit comes from the lane that holds it
  float a2[2] = {__bfloat162float(W[kB2 + lane]), __bfloat162float(W[kB2 + lane + 32])};
#pragma unroll 4
  for (int k = 0; k < kH; ++k) {
    const float hk = __shfl_sync(0xffffffffu, h1[k >> 5], k & 31);
    a2[0] = fmaf(__bfloat162float(W[kW2 + k * kH + lane]), hk, a2[0]);
    a2[1] = fmaf(__bfloat162float(W[kW2 + k * kH + lane + 32]), hk, a2[1]);
  }
  const float h2a = gelu_f(a2[0]), h2b = gelu_f(a2[1]);
  // layer 3: two sums over the warp
  float y0 = __bfloat162float(W[kW3 + lane]) * h2a + __bfloat162float(W[kW3 + lane + 32]) * h2b;
  float y1 = __bfloat162float(W[kW3 + kH + lane]) * h2a + __bfloat162float(W[kW3 + kH + lane + 32]) * h2b;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    y0 += __shfl_xor_sync(0xffffffffu, y0, o);
    y1 += __shfl_xor_sync(0xffffffffu, y1, o);
  }
  u0 = (y0 + __bfloat162float(W[kB3])) * nm[2 * kIn + 2] + nm[2 * kIn];
  u1 = (y1 + __bfloat162float(W[kB3 + 1])) * nm[2 * kIn + 3] + nm[2 * kIn + 1];
}

__device__ __forceinline__ void mark_pixel(uint32_t* bm, const int32_t* cpix, int64_t e) {
  const int32_t i = __ldg(cpix + e);
  if (i >= 0) atomicOr(bm + (i >> 5), 1u << (i & 31));
}

// Marks the kept entries of a group (out of line: few groups hold one).
__device__ __noinline__ void mark_group(uint32_t* bm, const int32_t* cpix, float4 v4, float thr, int64_t e) {
  const float xs[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
  for (int j = 0; j < 4; ++j)
    if (xs[j] > thr) mark_pixel(bm, cpix, e + j);
}

// The first clip interval [lo, hi] from plain FP32 totals of the full set
// about 0 (h: Omega, A1, OO, B1, B2; the formulas of finalise, poisson_sd
// and clip_step in single rounding); only the core is placed with it.
__device__ __forceinline__ void approx_interval(float n_set, const float (&h)[6], float k, int cutoff, int model,
                                                float dark, float& lo, float& hi, float& mu, float& sd) {
  lo = -FLT_MAX;
  hi = FLT_MAX;
  mu = sd = 0.0f;
  if (h[0] == 0.0f || h[2] == 0.0f) return;
  mu = __fdiv_rn(h[1], h[0]);
  const float vv = __fadd_rn(__fsub_rn(h[4], __fmul_rn(2.0f * mu, h[3])), __fmul_rn(__fmul_rn(mu, mu), h[2]));
  sd = vv > 0.0f ? __fsqrt_rn(__fdiv_rn(vv, h[2])) : 0.0f;
  if (model == SEP_ERROR_POISSON) {
    const float var = __fadd_rn(__fdiv_rn(h[3], h[2]), dark);
    sd = var > 0.0f ? __fsqrt_rn(var) : 0.0f;
  }
  if (cutoff == SEP_CUTOFF_CHAUVENET) {
    if (n_set <= 2.0f) return;
    k = chauvenet_k(n_set);
  }
  lo = __fsub_rn(mu, __fmul_rn(k, sd));
  hi = __fadd_rn(mu, __fmul_rn(k, sd));
}

// SURR 0: the plain method; 1: also record the surrogate's features and
// training targets; 2: place the first core from the surrogate's prediction
// of the final interval (the replay is the same exact loop).
template <int MODE, int PREC, int kWarps, int SURR>
__global__ void __launch_bounds__(32 * kWarps, kWarpsPerSM / kWarps) k_clip_warp(ClipArgs a) {
  constexpr bool KAHAN = PREC == SEP_PREC_KAHAN;
  // the tail's share of a step is merged over the lanes in FP32 except
  // where the per-lane sums are compensated (KAHAN) or merged in FP64
  constexpr int TPREC = PREC == SEP_PREC_DWORD ? SEP_PREC_PLAIN : PREC;
  constexpr int NF = Sums<MODE>::NF, NI = Sums<MODE>::NI;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // [a ring of kRing groups a lane for each warp (not with entry weights)]
  // [per warp its tail: 8-byte slots, slot k of lane l at 32 k + l]
  constexpr int kRingBytes = MODE == MODE_ENTRY ? 0 : kWarps * kRing * 512;
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(smem_raw) + (uint32_t)(warp * kRing * 512) + 16u * lane;
  uint2* tails = reinterpret_cast<uint2*>(smem_raw + kRingBytes);
  uint2* tail = tails + (size_t)warp * (32 * a.tcap) + lane;
  // with inference (SURR 2) the network's normalisation and BF16 weights
  // follow the tails, copied once per CTA (read by every item, they would
  // otherwise compete with the streamed rows for the L1 cache)
  float* nm_s = reinterpret_cast<float*>(tails + (size_t)kWarps * 32 * a.tcap);
  __nv_bfloat16* w_s = reinterpret_cast<__nv_bfloat16*>(nm_s + kNNorm);
  (void)w_s;
  if (SURR == 2) {
    for (int i = threadIdx.x; i < kNParams; i += 32 * kWarps) w_s[i] = a.mlp_w[i];
    for (int i = threadIdx.x; i < kNNorm; i += 32 * kWarps) nm_s[i] = __ldg(a.mlp_norm + i);
    __syncthreads();
  }

  // optional counters (added by lane 0 as they occur): items, pass B
  // scans, overflows, replay steps, tail entries listed, items marked from
  // the tail, full passes
  auto stat = [&](int i, unsigned v) {
    if (a.clip_stats && lane == 0 && v) atomicAdd(a.clip_stats + i, (unsigned long long)v);
  };
  unsigned long long su[2] = {0, 0};   // surrogate: items whose predicted core held / that re-placed it

  // Units of work: a bin of this launch (in the launch's order, longest rows
  // first) and a group of frames_per_cta frames, x fastest. A persistent
  // launch (a.queue set) sizes its grid to the resident CTAs and every CTA
  // takes the next unit from the queue counter until none is left; else
  // CTA (x, y) runs unit y * gridDim.x + x alone.
  __shared__ int unit_s;
  for (int it = 0;; ++it) {
    int unit;
    if (a.queue) {
      if (threadIdx.x == 0) unit_s = atomicAdd(a.queue, 1);
      __syncthreads();
      unit = unit_s;
    } else {
      unit = it == 0 ? (int)(blockIdx.y * gridDim.x + blockIdx.x) : a.units;
    }
    if (unit >= a.units) break;
    const int ux = unit % a.units_x;
    const int b = a.bin_list ? __ldg(a.bin_list + ux) : ux;
    const int f0 = (unit / a.units_x) * a.frames_per_cta;
    const int f1 = min(f0 + a.frames_per_cta, a.n_frames);
    const int r0 = __ldg(a.rowptr + b);
    const int n = __ldg(a.rowptr + b + 1) - r0;      // multiple of 4
    const int nq = n >> 2;
    // coefficient classes of the row; weight-0 carriers follow the last
    const int4 g4 = __ldg(reinterpret_cast<const int4*>(a.grp) + b);
    const ClassEnds ge{g4.x >> 2, g4.y >> 2, g4.z >> 2, g4.w >> 2};

    // (MODE_ENTRY) the row's weights, 0 on padding
    const float* wts = MODE == MODE_ENTRY ? a.w + r0 : nullptr;

    for (int f = f0 + warp; f < f1; f += kWarps) {
      // this item's values: entry e of the row at slot r0 + e of the staged frame
      const Row row{reinterpret_cast<const float4*>(a.stage + (int64_t)f * a.npos + r0)};
      const int64_t o = (a.orow ? a.orow[f] : (int64_t)f * a.nbins) + b;
      stat(0, 1);
      // ------------- pass A: where to place the core -------------
      float cLo, cHi, K;
      float pLo = 0.0f, pHi = 0.0f, pK = 0.0f;   // SURR 2: the plain placement, for a retry
      float feat[kIn], m1 = 0.0f, s1 = 0.0f;
      (void)feat;
      {
        float ss[NF], cz[NF];
        uint32_t ci[NI];
        // (rows of 2048 entries and more: every 4th group of 4, 512 and more:
        // every 2nd)
        const int step = nq >= 512 ? 4 : (nq >= 128 ? 2 : 1);
        lane_full_sums<MODE>(row, wts, ge, lane, step, ring, ss, ci);
#pragma unroll
        for (int v = 0; v < NF; ++v) cz[v] = 0.0f;
        float n_set, h[6], l[6], lo, hi, mu, sd;
        warp_totals<MODE, SEP_PREC_PLAIN>(ss, cz, ci, n_set, h, l);
        approx_interval(n_set * (float)step, h, a.k_clip, a.cutoff, a.error_model, a.dark_var, lo, hi, mu, sd);
        const float mg = __fmul_rn(kCoreMargin, sd);
        cLo = __fadd_rn(lo, mg);
        cHi = __fsub_rn(hi, mg);
        K = choose_shift(mu, sd);
        if (SURR != 0) {
          m1 = mu;
          s1 = sd;
          sample_features<MODE>(row, wts, ge, lane, step, n_set, h[0], m1, s1, feat);
        }
        if (SURR == 2) {
          // the predicted final interval, and the core half a deviation inside it
          pLo = cLo;
          pHi = cHi;
          pK = K;
          float u0, u1;
          warp_mlp(w_s, nm_s, feat, lane, u0, u1);
          const float mh = fmaf(s1, u0, m1), sh = s1 * expf(fminf(u1, 20.0f));
          if (s1 > 0.0f && sh > 0.0f && fabsf(mh) <= FLT_MAX && sh <= FLT_MAX) {
            const float half = __fmul_rn(a.k_clip, sh), mgs = __fmul_rn(kSurrMargin, sh);
            cLo = __fadd_rn(__fsub_rn(mh, half), mgs);
            cHi = __fsub_rn(__fadd_rn(mh, half), mgs);
          }
        }
      }
      // ------------- the loop of Eq. 19: replay on core + tail, or full passes -------------
      Bcast st;
      st.Ln = -FLT_MAX;
      st.Hn = FLT_MAX;
      st.L = -FLT_MAX;
      st.H = FLT_MAX;
      st.n_cur = -1.0f;
      st.steps = -1;
      st.done = 0;
      st.Kf = K;
      bool ovf = false, scan = true, retried = SURR != 2;
      int m = 0, scans = 0;
      float cn = 0.0f, ch[6], cl[6];
      for (;;) {
        const float Ln = st.Ln, Hn = st.Hn;
        if (scan) {
          // pass B: the core's sums and the tail, for the core placed last
          float ss[NF], cc[NF];
          uint32_t ci[NI];
          const bool fit =
              lane_core_sums<MODE, KAHAN>(row, wts, ge, lane, cLo, cHi, K, tail, a.tcap, ring, m, ss, cc, ci);
          ovf = __any_sync(0xffffffffu, !fit);
          ++scans;
          if (a.clip_stats) {
            const unsigned listed = __reduce_add_sync(0xffffffffu, (unsigned)m);
            stat(1, 1);
            stat(2, ovf ? 1 : 0);
            stat(4, listed);
          }
          if (!retried) {
            // first pass B only (the plain placement is inside the first
            // interval, not necessarily inside a later one): when the
            // predicted core left more entries outside it than the tail holds
            // (a heavy-tailed bin), the plain placement instead
            retried = true;
            if (ovf) {
              cLo = pLo;
              cHi = pHi;
              K = pK;
              continue;
            }
          }
          if (!ovf) warp_totals<MODE, PREC>(ss, cc, ci, cn, ch, cl);
          scan = false;
        }
        float n_set, h[6], l[6], Kf;
        if (!ovf) {
          // a step of the replay: the core sums plus the tail inside [Ln, Hn]
          float ts[5], tc[5], th[5], tl[5];
          uint32_t tn;
          lane_tail_sums<MODE, KAHAN>(tail, m, Ln, Hn, K, ts, tc, tn);
          tn = __reduce_add_sync(0xffffffffu, tn);
          stat(3, 1);
          n_set = cn + (float)tn;
#pragma unroll
          for (int v = 0; v < 6; ++v) h[v] = l[v] = 0.0f;
          if (st.steps < 0 || n_set != st.n_cur) {   // (an unchanged set ends the loop with the moments it has)
            tail_totals<MODE, TPREC>(ts, tc, tn, th, tl);
#pragma unroll
            for (int v = 0; v < 5; ++v) {
              h[v] = ch[v];
              l[v] = cl[v];
              if (MODE != MODE_ENTRY && (v == 0 || v == 2)) h[v] = __fadd_rn(h[v], th[v]);   // exact
              else add_pair<PREC>(h[v], l[v], th[v], tl[v]);
            }
          }
          Kf = K;
        } else {
          // a tail overflowed: a full pass over [Ln, Hn]
          float ss[NF], cc[NF];
          uint32_t ci[NI];
          Kf = st.Kf;
          lane_range_sums<MODE, KAHAN>(row, wts, ge, lane, Ln, Hn, Kf, ring, ss, cc, ci);
          stat(6, 1);
          warp_totals<MODE, PREC>(ss, cc, ci, n_set, h, l);
        }
        clip_step<PREC>(st, n_set, h, l, Kf, Ln, Hn, a.n_iter, a.k_clip, false, a.cutoff, a.error_model, a.dark_var);
        if (st.done) break;
        if (!ovf && (cLo < st.Ln || cHi > st.Hn)) {
          // the next interval cuts into the core: place it inside and scan again
          const float mg = __fmul_rn(kCoreMargin, st.sd);
          cLo = __fadd_rn(st.Ln, mg);
          cHi = __fsub_rn(st.Hn, mg);
          K = st.Kf;
          scan = true;
        }
      }
      if (lane == 0) {
        a.mean[o] = st.mu_hi;
        a.sigma[o] = st.sd;
        a.count[o] = (int32_t)st.n_cur;
        if (a.bounds) {
          a.bounds[2 * o] = st.L;
          a.bounds[2 * o + 1] = st.H;
        }
        if (a.iters) a.iters[o] = st.steps;
        if (SURR == 1) {
          // training record: the features and the result as normalised targets
          for (int k = 0; k < kIn; ++k) a.rec_feat[o * kIn + k] = feat[k];
          const bool ok = s1 > 0.0f && st.sd > 0.0f && st.n_cur >= 2.0f;
          a.rec_target[o * 2] = ok ? (st.mu_hi - m1) / s1 : __int_as_float(0x7fc00000);
          a.rec_target[o * 2 + 1] = ok ? logf(st.sd / s1) : __int_as_float(0x7fc00000);
        }
      }
      if (SURR == 2) su[(scans == 1 && !ovf) ? 0 : 1] += 1;
      // threshold of sparsification (Section 3) from the final state
      const float thr = pick_threshold<PREC>(st, a.k_pick);
      if (a.thr_out && lane == 0) a.thr_out[o] = thr;
      if (a.bitmap) {
        // kept pixels of this bin: its centre entries whose value exceeds the
        // threshold (only kept pixels touch the pixel table and the bitmap)
        uint32_t* bm = a.bitmap + (int64_t)f * a.words;
        const int32_t* cp = a.cpix + r0;
        // without an overflow and with thr at or above the core, no core entry
        // exceeds thr: the lane's tail, then the weight-0 carriers of the row;
        // else every entry (padding slots hold NaN, never above a threshold)
        if (MODE == MODE_ENTRY) {   // (no ring to list in: each lane marks its own)
          scan_row(row, 0, nq, lane, [&](const float4& v4, int q) {
            if (fmaxf(fmaxf(v4.x, v4.y), fmaxf(v4.z, v4.w)) > thr) mark_group(bm, cp, v4, thr, 4 * q);
          });
        } else {
          const bool from_tail = !ovf && thr >= cHi;
          if (from_tail) stat(5, 1);
          // The warp's kept entries are listed first (by ballots, in the idle
          // ring), then looked up a lane each, so the pixel loads of an item's
          // kept pixels are in flight together: with each lane looking up its
          // own, a warp waited for memory once a slot or two, a quarter of the
          // kernel's time.
          uint16_t* lst = reinterpret_cast<uint16_t*>(smem_raw) + warp * kMarkList;
          const uint32_t below = (1u << lane) - 1u;
          const int most = from_tail ? (int)__reduce_max_sync(0xffffffffu, m) : 0;
          int k = 0, q = from_tail ? ge.e3 : 0;
          while (k < most || q < nq) {
            int listed = 0;
#pragma unroll 1
            for (; k < most && listed <= kMarkList - 32; ++k) {
              uint2 t = make_uint2(0x7fc00000u, 0u);
              if (k < m) t = tail[32 * k];
              const bool kept = __uint_as_float(t.x) > thr;
              const uint32_t who = __ballot_sync(0xffffffffu, kept);
              if (kept) lst[listed + __popc(who & below)] = (uint16_t)t.y;
              listed += __popc(who);
            }
            if (k >= most) {
#pragma unroll 1
              for (; q < nq && listed <= kMarkList - 256; q += 64) {   // two groups a lane at a time
                float4 v[2];
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                  const float nan = __int_as_float(0x7fc00000);
                  v[u] = make_float4(nan, nan, nan, nan);
                  if (q + 32 * u + lane < nq) v[u] = __ldg(row.v4 + q + 32 * u + lane);
                }
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                  const float xs[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                  for (int j = 0; j < 4; ++j) {
                    const uint32_t who = __ballot_sync(0xffffffffu, xs[j] > thr);
                    if (xs[j] > thr) lst[listed + __popc(who & below)] = (uint16_t)(4 * (q + 32 * u + lane) + j);
                    listed += __popc(who);
                  }
                }
              }
            }
            __syncwarp();
#pragma unroll 1
            for (int i = lane; i < listed; i += 128) {
              int32_t px[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) px[u] = i + 32 * u < listed ? __ldg(cp + lst[i + 32 * u]) : -1;
#pragma unroll
              for (int u = 0; u < 4; ++u)
                if (px[u] >= 0) atomicOr(bm + (px[u] >> 5), 1u << (px[u] & 31));
            }
            __syncwarp();
          }
        }
      }
      __syncwarp();   // the tail is rewritten by the warp's next frame
    }
    // the next unit rewrites unit_s
    __syncthreads();
  }
  if (SURR == 2 && a.surr_stats && lane == 0) {
    if (su[0]) atomicAdd(a.surr_stats, su[0]);
    if (su[1]) atomicAdd(a.surr_stats + 1, su[1]);
  }
}

// Opt-in shared memory per block of the current device (cached).
int smem_optin() {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (cached[dev] == 0) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || v <= 0)
      v = 48 * 1024;
    cached[dev] = v;
  }
  return cached[dev];
}

// Multiprocessors of the current device (cached).
int sm_count() {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
  if (cached[dev] == 0) {
    int v = 0;
    if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) v = 1;
    cached[dev] = v;
  }
  return cached[dev];
}

// Shared memory of the surrogate's network in an inference launch.
constexpr long kNetBytes = kNNorm * 4 + ((kNParams * 2 + 15) & ~15);

// Tail slots a lane has. When its slots run out an item's remaining steps run
// as full passes, whose sums round differently, so the number is part of the
// results: it follows from the longest row and the plan's block size alone
// (what 1/12 of the row needs, at most what a block of that size had room for
// with a row's entry weights beside the tails), not from the launch's layout.
long clip_tail_cap(bool weights, int32_t cap, int warps, int surr) {
  const long wbytes = weights ? 4 * (((long)cap + 3) & ~3L) : 0;
  const long budget = (long)smem_optin() - kClipStaticSmem - wbytes - (surr == 2 ? kNetBytes : 0);
  long tcap = clip_tail_slots(cap, 32 * warps);
  if (warps * 256 * tcap > budget) tcap = std::max(0L, budget / (256L * warps));
  return tcap < 5 ? 0 : tcap;   // (no room for a tail: every step runs as a full pass)
}

// Shared memory of a launch: the warps' rings (not with entry weights) and tails.
size_t clip_launch_bytes(bool weights, int warps, long tcap, int surr) {
  return (size_t)(warps * ((weights ? 0 : kRing * 512) + 256 * tcap) + (surr == 2 ? kNetBytes : 0));
}

template <int MODE, int PREC, int kWarps, int SURR>
cudaError_t launch_warp_t(ClipArgs a, int n_ctas, long tcap, int mode, cudaStream_t s) {
  a.tcap = (int32_t)tcap;
  const size_t smem = clip_launch_bytes(MODE == MODE_ENTRY, kWarps, tcap, SURR);
  auto k = k_clip_warp<MODE, PREC, kWarps, SURR>;
  // resident CTAs per multiprocessor of this instance at this shared-memory
  // size, cached per device (the first query comes before any capture: the
  // attribute pass below asks it). A stale or missing value changes only the
  // grid of a persistent launch, never its results (0: not persistent).
  auto resident = [&]() -> int {
    static int occ_smem[64][8], occ_val[64][8] = {}, occ_next[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    for (int i = 0; i < 8; ++i)
      if (occ_val[dev][i] > 0 && occ_smem[dev][i] == (int)smem) return occ_val[dev][i];
    int v = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k, 32 * kWarps, smem) != cudaSuccess) v = 0;
    const int i = occ_next[dev]++ & 7;
    occ_smem[dev][i] = (int)smem;
    occ_val[dev][i] = v;
    return v;
  };
  if (mode != 2) {
    // the attribute only grows: size classes sharing this instance may set
    // it in any order before a capture
    static int attr[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) dev = 0;
    if ((int)smem > attr[dev]) {
      cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      attr[dev] = (int)smem;
    }
    if (mode == 1) {
      (void)resident();
      return cudaSuccess;
    }
  }
  const int gy = (a.n_frames + a.frames_per_cta - 1) / a.frames_per_cta;
  a.units_x = n_ctas;
  a.units = n_ctas * gy;
  dim3 grid(n_ctas, gy);
  if (a.queue) {
    // persistent: as many CTAs as stay resident, while the units outnumber them
    const int per_sm = resident();
    const int64_t slots = (int64_t)sm_count() * per_sm;
    if (per_sm > 0 && slots < a.units) {
      grid = dim3((unsigned)slots, 1);
      cudaError_t e = cudaMemsetAsync(a.queue, 0, sizeof(int32_t), s);
      if (e != cudaSuccess) return e;
    } else {
      a.queue = nullptr;
    }
  }
  k<<<grid, 32 * kWarps, smem, s>>>(a);
  return cudaGetLastError();
}

template <int MODE, int PREC, int SURR = 0>
cudaError_t launch_tail_b(const ClipArgs& a, int n_ctas, int tpb, int mode, cudaStream_t s) {
  int warps = tpb == 32 || tpb == 64 || tpb == 128 ? tpb / 32 : 8;
  const long tcap = clip_tail_cap(MODE == MODE_ENTRY, a.cap, warps, SURR);
  // the widest block up to the plan's whose rings and tails fit
  while (warps > 1 && clip_launch_bytes(MODE == MODE_ENTRY, warps, tcap, SURR) + kClipStaticSmem > (size_t)smem_optin())
    warps /= 2;
  switch (warps) {
    case 1: return launch_warp_t<MODE, PREC, 1, SURR>(a, n_ctas, tcap, mode, s);
    case 2: return launch_warp_t<MODE, PREC, 2, SURR>(a, n_ctas, tcap, mode, s);
    case 4: return launch_warp_t<MODE, PREC, 4, SURR>(a, n_ctas, tcap, mode, s);
    default: return launch_warp_t<MODE, PREC, 8, SURR>(a, n_ctas, tcap, mode, s);
  }
}

template <int MODE>
cudaError_t launch_p(const ClipArgs& a, int n_ctas, int tpb, int32_t prec, int mode, cudaStream_t s) {
  // the surrogate modes exist for the default precision only
  if (a.rec_feat) return launch_tail_b<MODE, SEP_PREC_DWORD, 1>(a, n_ctas, tpb, mode, s);
  // (inference: at least 4 warps a CTA share one copy of the weights)
  if (a.mlp_w) return launch_tail_b<MODE, SEP_PREC_DWORD, 2>(a, n_ctas, std::max(tpb, 128), mode, s);
  switch (prec) {
    case SEP_PREC_PLAIN: return launch_tail_b<MODE, SEP_PREC_PLAIN>(a, n_ctas, tpb, mode, s);
    case SEP_PREC_KAHAN: return launch_tail_b<MODE, SEP_PREC_KAHAN>(a, n_ctas, tpb, mode, s);
    case SEP_PREC_FP64MERGE: return launch_tail_b<MODE, SEP_PREC_FP64MERGE>(a, n_ctas, tpb, mode, s);
    default: return launch_tail_b<MODE, SEP_PREC_DWORD>(a, n_ctas, tpb, mode, s);
  }
}

}  // namespace

size_t clip_smem_bytes(int32_t cap, bool weighted) {
  // what clip_tail_cap takes from the tails' budget for a row's entry weights
  // (read through the caches, they need no shared memory themselves)
  size_t smem = weighted ? (size_t)cap * 4 : 0;
  return (smem + 15) & ~(size_t)15;
}

int32_t clip_tail_slots(int32_t cap, int32_t tpb) {
  // per lane of a warp: 1/12 of the row over 32 lanes (a tail holds about
  // 1/20 of a row's entries), plus the 4 slots a pass B keeps free and some
  // room for uneven lanes; a lane that runs out switches its item to full
  // passes (tpb: the block size, one warp per item whatever it is)
  (void)tpb;
  return (int32_t)((cap + 383) / 384) + 6;
}

cudaError_t launch_integrate_clip(const ClipArgs& a, int n_ctas, int tpb, bool split, bool has_norm,
                                  int32_t precision, int mode, cudaStream_t s) {
  if (a.n_frames <= 0 || n_ctas <= 0) return cudaSuccess;
  if (has_norm) return launch_p<MODE_ENTRY>(a, n_ctas, tpb, precision, mode, s);
  return split ? launch_p<MODE_CLASS>(a, n_ctas, tpb, precision, mode, s)
               : launch_p<MODE_UNIT>(a, n_ctas, tpb, precision, mode, s);
}

}  // namespace sep
