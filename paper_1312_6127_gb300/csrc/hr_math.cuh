// FP64 reciprocal, square root and reciprocal square root for the hot kernels.
//
// Those kernels are bound by the number of FP64 instructions (each holds an
// SM's FP64 pipe for 16 clocks), and a division or square root of the
// language costs about ten.  Here the hardware's reciprocal (square root) seed
// (PTX rcp.approx.ftz.f64, rsqrt.approx.ftz.f64: about 20 bits, computed off the
// FP64 pipe) takes one step of the cubically convergent iteration for 1/x
// (y (1 + e + e^2), e = 1 - x y) or 1/sqrt(x) (y (1 + e/2 + 3 e^2/8),
// e = 1 - x y^2; Householder's family), which leaves e^3 and 5 e^3/16 of
// truncation, 2^-60 and 2^-58.7 for |e| of 2^-20 and 2^-19: below the rounding of
// the last operation (sqrt(x) = x y + x y q with one rounding of the sum, y q the
// correction).  1/x costs 3 FP64 instructions, 1/sqrt(x) 5, sqrt(x) 7, both
// together 8.  Largest errors over a million arguments of every exponent, against
// extended precision: 1/x 0.504 ulp, 1/sqrt(x) 0.505, sqrt(x) 0.515.  Arguments
// outside the range where the seed and the residual are normal numbers (zero,
// subnormal, infinite, NaN, negative under the root, above 2^1022) go to the
// language's operation.
#pragma once
#include <cuda_runtime.h>

namespace hr {

static __device__ __noinline__ double rcp_any(double x) { return 1.0 / x; }
static __device__ __noinline__ double sqrt_any(double x) { return ::sqrt(x); }
static __device__ __noinline__ double rsqrt_any(double x) { return 1.0 / ::sqrt(x); }

// biased exponent of the high word between 1 and 2044
__device__ __forceinline__ bool seed_range(int hi) { return (unsigned)(hi - 0x00100000) < 0x7fc00000u; }

__device__ __forceinline__ double rcp(double x) {
  if (!seed_range(__double2hiint(x) & 0x7fffffff)) return rcp_any(x);
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// The seed y of 1/sqrt(x) with its correction q: 1/sqrt(x) = y + y q.
__device__ __forceinline__ double rsqrt_seed(double x, double* q) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = __hiloint2double(__double2hiint(y), 0);  // 21 bits: y^2 is exact
  const double e = fma(-x, y * y, 1.0);
  *q = e * fma(e, 0.375, 0.5);
  return y;
}
__device__ __forceinline__ double rsqrt64(double x) {
  if (!seed_range(__double2hiint(x))) return rsqrt_any(x);
  double q;
  const double y = rsqrt_seed(x, &q);
  return fma(y, q, y);
}
// sqrt(x), and 1/sqrt(x) in *r
__device__ __forceinline__ double sqrt_rsqrt(double x, double* r) {
  if (!seed_range(__double2hiint(x))) {
    *r = rsqrt_any(x);
    return sqrt_any(x);
  }
  double q;
  const double y = rsqrt_seed(x, &q), c = y * q;
  *r = y + c;
  return fma(x, y, x * c);
}
__device__ __forceinline__ double sqrt64(double x) {
  if (!seed_range(__double2hiint(x))) return sqrt_any(x);
  double q;
  const double y = rsqrt_seed(x, &q);
  return fma(x, y, x * (y * q));
}

// FP64 <-> FP32 with the bits of the language's conversions, by integer
// operations: the hardware's conversion is an FP64 pipe instruction like any
// other, and a zone's FP32 Jacobian takes about fifty.  Numbers beyond the normal
// FP32 range go to the language's conversion.
static __device__ __noinline__ float narrow_any(double x) { return (float)x; }
static __device__ __noinline__ double widen_any(float x) { return (double)x; }

__device__ __forceinline__ float narrow(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  if ((hi & 0x7ff00000u) - (897u << 20) >= (254u << 20))
    return ((hi << 1) | lo) == 0 ? __uint_as_float(hi) : narrow_any(x);
  // round to nearest even at bit 29; the exponent's bias 1023 -> 127
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) + 0x0fffffffu + ((lo >> 29) & 1u);
  return __uint_as_float(((unsigned)(b >> 29) - (896u << 23)) | (hi & 0x80000000u));
}

__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x);
  if ((u & 0x7f800000u) - 0x00800000u >= 0x7f000000u)
    return (u << 1) == 0 ? __hiloint2double((int)u, 0) : widen_any(x);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + (896u << 20))), (int)(u << 29));
}

}  // namespace hr
