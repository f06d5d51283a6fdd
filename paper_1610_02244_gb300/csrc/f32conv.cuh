// Conversions between FP64 and FP32 by integer operations on the IEEE-754 layouts, for the
// FP32-arithmetic passes over FP64 vectors: on GB300 an SM retires two FP64 operations per
// clock, and these keep the element loops off the FP64 pipe.
//   f32_of: truncation toward zero to 23 mantissa bits; magnitudes below 2^-126 become a
//           signed zero, magnitudes of 2^128 and above (and non-finite values) infinity.
//   f64_of: exact; FP32 subnormals become a signed zero.
//   fixed54: the fixed-point form floor(|v| 2^(54 - esc)) of |v| < 2^esc.
// The same code compiles for the host, where tests/f32conv_host.cu checks it against the
// C library's conversions.
#pragma once
#include <cstdint>
#include <cstring>

#include <cuda_runtime.h>

namespace tnt {

__host__ __device__ __forceinline__ uint64_t bits_of(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  std::memcpy(&u, &x, sizeof u);
  return u;
#endif
}
__host__ __device__ __forceinline__ double double_of_bits(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  std::memcpy(&x, &u, sizeof x);
  return x;
#endif
}
__host__ __device__ __forceinline__ unsigned bits_of(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  unsigned u;
  std::memcpy(&u, &x, sizeof u);
  return u;
#endif
}
__host__ __device__ __forceinline__ float float_of_bits(unsigned u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float x;
  std::memcpy(&x, &u, sizeof x);
  return x;
#endif
}

__host__ __device__ __forceinline__ float f32_of(double x) {
  const uint64_t u = bits_of(x);
  const unsigned hi = (unsigned)(u >> 32);
  const unsigned e = (hi >> 20) & 0x7ffu, sgn = hi & 0x80000000u;
  const unsigned m = (unsigned)(u >> 29) & 0x7fffffu;  // the 23 leading mantissa bits
  unsigned b = sgn | ((e - 896u) << 23) | m;           // exponent bias 1023 -> 127
  b = (e <= 896u) ? sgn : b;
  b = (e >= 1151u) ? (sgn | 0x7f800000u) : b;
  return float_of_bits(b);
}

__host__ __device__ __forceinline__ double f64_of(float f) {
  const unsigned b = bits_of(f);
  const unsigned e = (b >> 23) & 0xffu, sgn = b & 0x80000000u, m = b & 0x7fffffu;
  unsigned hi = sgn | ((e + 896u) << 20) | (m >> 3), lo = m << 29;
  if (e == 0u) {
    hi = sgn;
    lo = 0u;
  }
  if (e == 255u) hi = sgn | 0x7ff00000u | (m >> 3);
  return double_of_bits(((uint64_t)hi << 32) | lo);
}

// F = floor(|v| 2^(54 - esc)) for |v| < 2^esc: the 53-bit mantissa shifted (exact).  Only its host
// check uses it now; the slices of the FP64-accurate GEMM come from oz_fixed (oz.cuh).
__host__ __device__ __forceinline__ uint64_t fixed54(double v, int esc) {
  const uint64_t u = bits_of(v);
  const int eb = (int)((u >> 52) & 0x7ff);
  uint64_t mant = u & ((1ull << 52) - 1);
  if (eb) mant |= 1ull << 52;
  const int sh = (eb ? eb : 1) - 1021 - esc;  // F = mant 2^sh, F < 2^54
  if (sh >= 0) return mant << sh;
  return sh <= -64 ? 0ull : mant >> (-sh);
}

#ifdef __CUDACC__
// 1 / sqrt(s) for normal positive s and 1 / d for normal d, |d| < 2^923, from an FP32 seed (relative
// error below 2^-21) by one step of third order: Householder's iteration for s y^2 = 1 (A. S.
// Householder, The Numerical Treatment of a Single Nonlinear Equation, 1970),
// y (1 + e/2 + 3/8 e^2) with e = 1 - s y^2, and the hyperpower iteration (M. Altman, Pacific J.
// Math. 10, 1960), r (1 + e + e^2) with e = 1 - d r.  The series' rest is of order e^3 = 2^-60.
// Rounding: the reciprocal's e is exact to its own last bit, so that one rounding, 2^-53,
// is left; the root's e carries the rounding of s y, in all 1.5 2^-53, against 2 2^-53 of
// 1.0 / sqrt(s) (tests/newton_gpu.cu).  The arguments are scaled to [1, 4) and [1, 2) by exponent
// arithmetic.
__device__ __forceinline__ double rsqrt_newton(double s) {
  const int hi = __double2hiint(s), ex = (hi >> 20) - 1023, h = ex >> 1;
  const double m = __hiloint2double((hi & 0xfffff) | ((1023 + (ex & 1)) << 20), __double2loint(s));
  float y0;
  asm("rsqrt.approx.f32 %0, %1;" : "=f"(y0) : "f"(f32_of(m)));
  const double y = f64_of(y0);
  const double e = fma(-m * y, y, 1.0);
  const double r = fma(y, e * fma(e, 0.375, 0.5), y);
  return __hiloint2double(__double2hiint(r) - (h << 20), __double2loint(r));
}
__device__ __forceinline__ double rcp_newton(double d) {
  const int hi = __double2hiint(d), ex = ((hi >> 20) & 0x7ff) - 1023;
  const double m = __hiloint2double((hi & 0x800fffff) | (1023 << 20), __double2loint(d));
  float r0;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r0) : "f"(f32_of(m)));
  const double r = f64_of(r0);
  const double e = fma(-m, r, 1.0);
  const double q = fma(r, fma(e, e, e), r);
  return __hiloint2double(__double2hiint(q) - (ex << 20), __double2loint(q));
}

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
#endif

}  // namespace tnt
