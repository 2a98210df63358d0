// The round-to-nearest code of one weight (paper: Eq. 2).
//
// The code is the fp64 rounding of (w - b) / a, half to even, clamped to the grid.  The fp32 quotient is off by at most
// 3 * 2^-24 of itself (6 * 2^-24 where the inverse of the scale is subnormal), 1e-4 where it is within 256 levels, so
// unless it lies within 2e-4 of the middle between two levels both round to the same level; the one in 2500 that does is
// decided in fp64, and so is a quotient that is none or overflows (groups that span more than 3.4e38).
#pragma once

#include "common.cuh"

namespace cdq {

// 1 / a for rtn_code; a scale whose inverse overflows gives a NaN, with which every code is decided in fp64.
__device__ __forceinline__ float rtn_inverse(float a) {
  const float inv = 1.0f / a;
  return inv <= 3.4e38f ? inv : __int_as_float(0x7FFFFFFF);
}
// The code by an fp64 division (kept out of line: it runs once in 2500 weights).
static __device__ __noinline__ unsigned rtn_code_f64(float w, float a, float b, float top) {
  double q = rint(__ddiv_rn(__dadd_rn((double)w, -(double)b), (double)a));
  q = q < 0.0 ? 0.0 : q;
  q = q > (double)top ? (double)top : q;
  return (unsigned)(unsigned char)q;
}
// a > 0; top: the highest level
__device__ __forceinline__ unsigned rtn_code(float w, float a, float inv_a, float b, float top) {
  constexpr float kMagic = 12582912.0f;   // 1.5 * 2^23: adding it rounds to an integer, to the even one in the middle
  const float t = (w - b) * inv_a;
  const float c = fminf(fmaxf(t, 0.f), top);
  const float m = c + kMagic;
  if (!(fabsf(c - (m - kMagic)) < 0.4998f) || !(fabsf(t) <= 3.402823466e38f)) return rtn_code_f64(w, a, b, top);
  return __float_as_uint(m) & 255u;
}

}  // namespace cdq
