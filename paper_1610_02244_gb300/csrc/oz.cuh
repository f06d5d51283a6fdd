// Integer pieces of the FP64-accurate GEMM (oz.cu): digits of an FP64 value, and the FP64
// value of a combined level sum.  The same code compiles for the host, where
// tests/oz_host.cu checks it.
#pragma once
#include "f32conv.cuh"

namespace tnt {

// F = |v| 2^(55 - a) rounded to nearest, a = e - 1022 the exponent of a power of two above
// |v|: e is the largest biased exponent of the row (its maximum is below 2^(e - 1022)).
// F <= 2^55; a row of zeros and subnormals (e = 0) uses the exponent of e = 1.
__host__ __device__ __forceinline__ uint64_t oz_fixed(double v, int e) {
  const uint64_t u = bits_of(v);
  const int eb = (int)((u >> 52) & 0x7ff);
  uint64_t m = u & ((1ull << 52) - 1);
  if (eb) m |= 1ull << 52;
  const int sh = (eb ? eb : 1) + 2 - (e ? e : 1);  // <= 2
  if (sh >= 0) return m << (sh & 3);
  return sh <= -55 ? 0ull : (m + (1ull << (-sh - 1))) >> (-sh);
}

// F = sum_p d_p 128^(7-p) with d_0 in [0, 64] and the others in [-64, 63]: adding 64 at
// each lower place (G = F + OZ_BIAS) makes them the plain base-128 digits of G
constexpr uint64_t OZ_BIAS = 64ull * ((1ull << 0) + (1ull << 7) + (1ull << 14) + (1ull << 21) + (1ull << 28) +
                                      (1ull << 35) + (1ull << 42));
// signs of two values as bits 15 and 31
__host__ __device__ __forceinline__ uint32_t oz_signs(double a, double b) {
  return ((uint32_t)(bits_of(a) >> 48) & 0x8000u) | ((uint32_t)(bits_of(b) >> 32) & 0x80000000u);
}
// digits p (0 the highest) of two biased values as an FP16 pair, negated where sgn's bits 15
// and 31 say so.  0x6400 + u is the FP16 number 1024 + u, so one packed subtraction of
// 1024 (+ 64) makes both digits, exactly.
__host__ __device__ __forceinline__ uint32_t oz_digit2(uint64_t G0, uint64_t G1, int p, uint32_t sgn) {
  const uint32_t m = p == 0 ? 0x7fffu : 0x7fu;
  const int s = 7 * (7 - p);
  const uint32_t w = ((uint32_t)(G0 >> s) & m) | (((uint32_t)(G1 >> s) & m) << 16) | 0x64006400u;
#ifdef __CUDA_ARCH__
  const uint32_t o = p == 0 ? 0xe400e400u : 0xe440e440u;  // -1024, -1088
  uint32_t r;
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(w), "r"(o));
  return r ^ sgn;
#else
  uint32_t r = 0;
  for (int t = 0; t < 2; ++t) {
    const int d = (int)((w >> (16 * t)) & 0x3ffu) - (p == 0 ? 0 : 64);
    uint32_t h = 0;
    if (d) {
      int a = d < 0 ? -d : d, ex = 0;
      while ((a >> (ex + 1)) != 0) ++ex;
      h = (d < 0 ? 0x8000u : 0u) | ((uint32_t)(15 + ex) << 10) | (uint32_t)((a << (10 - ex)) & 0x3ff);
    }
    r |= h << (16 * t);
  }
  return r ^ sgn;
#endif
}

__host__ __device__ __forceinline__ int oz_clz(uint32_t x) {
#ifdef __CUDA_ARCH__
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}

// m 2^(e - 1086) rounded to nearest even for e < 1 (subnormal) or e > 2046 (infinity); bit
// 63 of m is set, its bit 0 is sticky
__host__ __device__ __noinline__ inline uint64_t oz_round_edge(uint64_t m, int e) {
  if (e > 2046) return 0x7ff0000000000000ull;
  const int sh = 12 - e;  // one more place per step below e = 1
  if (sh >= 65) return 0;
  const uint64_t q = sh == 64 ? 0ull : m >> sh, half = 1ull << (sh - 1);
  const uint64_t rest = sh == 64 ? m : m & ((1ull << sh) - 1);
  return q + ((rest > half) | ((rest == half) & (q & 1ull)));
}

// (2^28 H + L) 2^(ea + eb - 2105), rounded to nearest even (ea, eb: the row's and the
// column's exponent fields; 2 (-1022) - 61 = -2105).  A field of 2047 marks an infinity or
// NaN in the row or column: NaN.  |2^28 H + L| < 2^95.  About 40 integer instructions on
// 32-bit words, without a branch in the normal range (a 128-bit form with branches took
// 430 clocks per value and more time than the MMAs).
__host__ __device__ __forceinline__ double oz_value(long long H, long long L, int ea, int eb) {
  const uint64_t h = (uint64_t)H << 28;
  uint64_t lo = h + (uint64_t)L;
  uint32_t top = (uint32_t)(H >> 36) + (uint32_t)(L >> 63) + (uint32_t)(lo < h);
  const uint32_t neg = (uint32_t)((int32_t)top >> 31);
  lo = (lo ^ (uint64_t)(int64_t)(int32_t)neg) + (neg & 1u);
  top = (top ^ neg) + (neg & (uint32_t)(lo == 0));
  // the leading word to a2, its leading one to bit 31
  uint32_t a2 = top, a1 = (uint32_t)(lo >> 32), a0 = (uint32_t)lo;
  int sh = 0;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const bool z0 = a2 == 0;
    a2 = z0 ? a1 : a2;
    a1 = z0 ? a0 : a1;
    a0 = z0 ? 0u : a0;
    sh += z0 ? 32 : 0;
  }
  const int c = oz_clz(a2);
  if (a2 == 0) return ea == 2047 || eb == 2047 ? double_of_bits(0x7ff8000000000000ull) : 0.0;
#ifdef __CUDA_ARCH__
  const uint32_t mh = __funnelshift_l(a1, a2, c), ml = __funnelshift_l(a0, a1, c) | (uint32_t)((a0 << c) != 0);
#else
  const uint32_t mh = c ? (a2 << c) | (a1 >> (32 - c)) : a2,
                 ml = (c ? (a1 << c) | (a0 >> (32 - c)) : a1) | (uint32_t)((a0 << c) != 0);
#endif
  const uint64_t m = ((uint64_t)mh << 32) | ml;
  const int e = 95 - sh - c + (ea ? ea : 1) + (eb ? eb : 1) - 2105 + 1023;  // biased exponent
  const uint64_t s = (uint64_t)(neg & 0x80000000u) << 32;
  if (ea == 2047 || eb == 2047) return double_of_bits(0x7ff8000000000000ull);
  if ((unsigned)(e - 1) >= 2046u) return double_of_bits(s | oz_round_edge(m, e));
  const uint32_t up = ((ml & 0x7ffu) + 0x3ffu + ((ml >> 11) & 1u)) >> 11;
  // the leading one adds one to the exponent field, and so does a carry out of the mantissa
  return double_of_bits(s | (((uint64_t)(unsigned)(e - 1) << 52) + (m >> 11) + up));
}

}  // namespace tnt
