// FP64 helpers that spare GB300's FP64 pipe (device code): a conversion between
// FP32 and FP64 costs the pipe as much as a multiplication, and a division ten
// times that.
#pragma once

#include <cuda_runtime.h>

namespace ebb {

// An FP32 value in FP64, exactly, by integer instructions: zero and normal
// values; the others take the conversion.
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
  if (m == 0u) return __hiloint2double((int)u, 0);
  return (double)x;
}

// The FP32 value of x (round to nearest even), likewise: results in FP32's normal
// range and zero; the others take the conversion.
__device__ __forceinline__ float narrow(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned m = hi & 0x7fffffffu;
  if (m - 0x38100000u < 0x0fd00000u) {   // 2^-126 <= |x| < 2^127
    const unsigned t = ((m - 0x38000000u) << 3) | (lo >> 29), rest = lo << 3;   // kept bits, dropped bits
    const unsigned up = rest > 0x80000000u || (rest == 0x80000000u && (t & 1u)) ? 1u : 0u;
    return __uint_as_float((hi & 0x80000000u) | (t + up));
  }
  if ((m | lo) == 0u) return __uint_as_float(hi);
  return (float)x;
}

// The same for a value of either precision.
__device__ __forceinline__ double to_f64(float x) { return widen(x); }
__device__ __forceinline__ double to_f64(double x) { return x; }

// 1 / x to within about an ulp: Newton's iteration r += r (1 - x r) twice from an
// FP32 reciprocal (relative errors 2^-23, 2^-46, rounding); values outside
// FP32's range take the division.
__device__ __forceinline__ double recip(double x) {
  const unsigned m = (unsigned)__double2hiint(x) & 0x7fffffffu;
  if (m - 0x38500000u >= 0x0f400000u) return 1.0 / x;   // not in 2^-122 .. 2^122
  double r = widen(__frcp_rn(narrow(x)));
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}

}  // namespace ebb
