// Host check of csrc/oz.cuh, the integer pieces of the FP64-accurate GEMM: the digits of a
// value must add up to its 55-bit fixed-point form rounded to nearest, with every digit in
// the range the exactness bound assumes; oz_value must be the correctly rounded FP64 value
// of (2^28 H + L) 2^(ea + eb - 2105), through the subnormal range and overflow.  Prints the
// number of mismatches and exits non-zero on any.
#include <cmath>
#include <cstdio>

#include "oz.cuh"

static uint64_t rng_state = 0x9e3779b97f4a7c15ull;
static uint64_t next_u64() {  // splitmix64
  uint64_t z = (rng_state += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

static int half_int(unsigned h) {  // an FP16 integer
  if (!(h & 0x7fffu)) return 0;
  const double v = std::ldexp(1.0 + (double)(h & 0x3ffu) / 1024.0, (int)((h >> 10) & 31u) - 15);
  return (int)((h & 0x8000u) ? -v : v);
}

// |v| 2^55 / 2^(e - 1022) by scaling in two exact steps, rounded half up
static int check_digits(double v, int e) {
  const uint64_t F = tnt::oz_fixed(v, e);
  const int a = (e ? e : 1) - 1022;
  // |v| = m 2^x exactly; F = m 2^(x + 55 - a), halves up
  int x;
  const double f = std::frexp(std::fabs(v), &x);
  unsigned __int128 m = (unsigned __int128)(uint64_t)std::ldexp(f, 53);
  const int sh = x - 53 + 55 - a;
  uint64_t want;
  if (sh >= 0) want = (uint64_t)(m << sh);
  else if (sh < -60) want = 0;
  else want = (uint64_t)((m + ((unsigned __int128)1 << (-sh - 1))) >> -sh);
  int bad = F != want;
  long long sum = 0;
  for (int p = 0; p < 8; ++p) {
    const unsigned w = tnt::oz_digit2(F + tnt::OZ_BIAS, F + tnt::OZ_BIAS, p, tnt::oz_signs(1.0, -1.0));
    const int d = half_int(w & 0xffffu);
    bad |= p == 0 ? (d < 0 || d > 64) : (d < -64 || d > 63);
    bad |= half_int(w >> 16) != -d;
    sum = sum * 128 + d;
  }
  bad |= (uint64_t)sum != F;
  if (bad) std::printf("digits of %.17g (field %d): F %llu, expected %llu, sum %lld\n", v, e,
                       (unsigned long long)F, (unsigned long long)want, sum);
  return bad;
}

static int check_value(long long H, long long L, int ea, int eb) {
  const double got = tnt::oz_value(H, L, ea, eb);
  const __int128 T = (__int128)H * ((__int128)1 << 28) + L;
  const int x = (ea ? ea : 1) + (eb ? eb : 1) - 2105;
  // round |T| 2^x to a double by hand: keep the bits a double of that size has
  unsigned __int128 m = T < 0 ? -(unsigned __int128)T : (unsigned __int128)T;
  double want = 0;
  if (m) {
    int top = 127;
    while (!((m >> top) & 1)) --top;
    int drop = top - 52;                          // bits below the last kept one
    if (top + x < -1022) drop += -1022 - (top + x);
    if (drop > 0) {
      if (drop > 126) m = 0;
      else {
        const unsigned __int128 rest = m & (((unsigned __int128)1 << drop) - 1), half = (unsigned __int128)1 << (drop - 1);
        m >>= drop;
        if (rest > half || (rest == half && (m & 1))) ++m;
      }
    } else drop = 0;
    want = std::ldexp((double)(uint64_t)m, drop + x);
    if (T < 0) want = -want;
  }
  if (want == 0) return got == 0 ? 0 : (std::printf("value %g, expected 0\n", got), 1);
  if (tnt::bits_of(got) != tnt::bits_of(want)) {
    std::printf("value of %lld, %lld, %d, %d: %.17g, expected %.17g\n", H, L, ea, eb, got, want);
    return 1;
  }
  return 0;
}

int main() {
  int bad = 0;
  for (int i = 0; i < 300000; ++i) {  // entries up to 60 binades below their row's maximum
    const uint64_t r = next_u64();
    const int e = 70 + (int)(next_u64() % 1900), eb = e - (int)(next_u64() % 62);
    const double v = tnt::double_of_bits(((uint64_t)eb << 52) | (r >> 12));
    bad += check_digits((r & 1) ? -v : v, e);
  }
  bad += check_digits(0.0, 0) + check_digits(4.9e-324, 0) + check_digits(4.9e-324, 1) + check_digits(1.0, 1023) +
         check_digits(std::nextafter(2.0, 0.0), 1023) + check_digits(std::nextafter(1.0, 0.0), 1022);
  for (int i = 0; i < 600000; ++i) {
    const int s = (int)(next_u64() % 48), t = (int)(next_u64() % 52);
    const long long H = (long long)(next_u64() >> 13) >> s, L = (long long)(next_u64() >> 11) >> t;
    const int ea = 1 + (int)(next_u64() % 2046);
    const int eb = i % 3 == 0 ? 1 + (int)(next_u64() % 2046) : std::min(2046, std::max(1, 2046 - ea + (int)(next_u64() % 60) - 30));
    bad += check_value((i & 1) ? -H : H, (i & 2) ? -L : L, ea, eb);
  }
  for (long long H : {0ll, 1ll, -1ll, (1ll << 52), -(1ll << 52)})
    for (long long L : {0ll, 1ll, -1ll, (1ll << 27), -(1ll << 28), (1ll << 53) - 1, -(1ll << 53)})
      for (int ea : {0, 1, 500, 1023, 2046})
        for (int eb : {0, 1, 600, 1023, 1100, 2046}) bad += check_value(H, L, ea, eb);
  bad += !std::isnan(tnt::oz_value(1, 1, 2047, 3)) + !std::isnan(tnt::oz_value(0, 0, 3, 2047));
  std::printf("mismatches %d\n", bad);
  return bad ? 1 : 0;
}
