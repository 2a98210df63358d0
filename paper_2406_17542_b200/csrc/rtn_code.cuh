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
// Four neighbouring codes as bytes (a <= 0: code 0).  One branch for the four (with one for each, and the bytes put together by shifts, the
// codes of 14336 x 16384 weights took a quarter longer;
// min, max and a sum that keeps a NaN instead of a chain of conditions: 341 -> 287 us for grid and codes of them in groups of 128).
__device__ __forceinline__ float rtn_inverse_or_zero(float a) { return a > 0.f ? rtn_inverse(a) : 0.f; }
__device__ __forceinline__ unsigned rtn_code4(const float (&w)[4], const float (&a)[4], const float (&inv_a)[4], const float (&b)[4],
                                              float top) {
  constexpr float kMagic = 12582912.0f;
  unsigned m[4];
  float off = 0.f, not_finite = 0.f;   // the largest distance from a level; a NaN if a quotient is none or overflows
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const float t = (w[v] - b[v]) * inv_a[v];
    const float c = fminf(fmaxf(t, 0.f), top);
    const float r = c + kMagic;
    off = fmaxf(off, fabsf(c - (r - kMagic)));
    not_finite = fmaf(t, 0.f, not_finite);
    m[v] = __float_as_uint(r);
  }
  if (!(off < 0.4998f && not_finite == 0.f)) {
    unsigned q = 0u;
#pragma unroll
    for (int v = 0; v < 4; ++v) q |= (a[v] > 0.f ? rtn_code(w[v], a[v], inv_a[v], b[v], top) : 0u) << (8 * v);
    return q;
  }
  return __byte_perm(__byte_perm(m[0], m[1], 0x0040), __byte_perm(m[2], m[3], 0x0040), 0x5410);
}

}  // namespace cdq
