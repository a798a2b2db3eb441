// Device helpers shared by the libsep kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "sep.h"

namespace sep {

// Corrected value of pixel `col` of one frame (Section 1.2 and Eq. 1).
// Raw Jungfrau words: the two top bits select the gain level (code 0 -> 0,
// code 1 -> 1, codes 2 and 3 -> 2) and the low 14 bits are the ADC value;
// photons = RN32(RN32(adc - pedestal) / gain), IEEE round-to-nearest without
// fused or approximate operations. A per-pixel norm divides the result.
template <int DT, bool NORM>
__device__ __forceinline__ float pixel_value(const void* frame, int64_t col, int64_t npix, const float* ped,
                                             const float* gain, const float* norm) {
  float p;
  if (DT == SEP_DTYPE_U16_JF) {
    uint32_t u = __ldg(reinterpret_cast<const uint16_t*>(frame) + col);
    uint32_t code = u >> 14;
    int64_t lvl = code == 0 ? 0 : (code == 1 ? 1 : 2);
    float adc = (float)(u & 0x3FFFu);
    float x = __fsub_rn(adc, __ldg(ped + lvl * npix + col));
    p = __fdiv_rn(x, __ldg(gain + lvl * npix + col));
  } else {
    p = __ldg(reinterpret_cast<const float*>(frame) + col);
  }
  if (NORM) p = __fdiv_rn(p, __ldg(norm + col));
  return p;
}

// Level-0 calibration of one pixel, for threads that correct the same pixel
// of many frames: the pedestal, the gain, r = RN(1 / gain), and the words
// that value() takes, those below limit (2^14: level 0; 0 where gain or
// pedestal lie outside the range its correction step is exact in). The other
// words go through pixel_value().
//
// RN((adc - ped) / gain) needs no division: with d = RN(adc - ped) and
// q = RN(d r), the residual e = d - q gain is exact under a fused
// multiply-add, and RN(q + e r) is the correctly rounded quotient
// (Markstein's correction, IBM J. Res. Dev. 34(1), 1990) as long as gain,
// quotient and residual are normal: with the ranges below a d other than 0
// lies between 2^-83 and 2^61 (the spacing of the larger of adc and ped
// bounds it below) and q between 2^-124 and 2^102; d = 0 gives the
// quotient's zero.
struct Level0 {
  float ped = 0.0f, gain = 1.0f, r = 1.0f;
  uint32_t limit = 0;
  __device__ __forceinline__ void set(float p, float g) {
    ped = p;
    gain = g;
    r = __frcp_rn(g);
    const float ag = fabsf(g), ap = fabsf(p);
    limit = ag >= 0x1p-40f && ag <= 0x1p40f && (p == 0.0f || (ap >= 0x1p-60f && ap <= 0x1p60f)) ? 0x4000u : 0u;
  }
  __device__ __forceinline__ float value(uint32_t u) const { return value_of((float)u); }
  __device__ __forceinline__ float value_of(float adc) const {
    const float d = __fsub_rn(adc, ped);
    const float q = __fmul_rn(d, r);
    return __fmaf_rn(__fmaf_rn(-q, gain, d), r, q);
  }
};

template <int DT>
__device__ __forceinline__ const void* frame_ptr(const void* frames, int64_t f, int64_t npix) {
  if (DT == SEP_DTYPE_U16_JF) return reinterpret_cast<const uint16_t*>(frames) + f * npix;
  return reinterpret_cast<const float*>(frames) + f * npix;
}

}  // namespace sep
