// Device check of rsqrt_newton and rcp_newton (csrc/f32conv.cuh).  On [1, 4) and [1, 2): relative errors
// from residuals computed in two doubles, over random mantissas and those next to the ends.
// Over all exponents that the callers admit, and both signs: the same bits, scaled.
#include <cstdint>
#include <cstdio>

#include "f32conv.cuh"

using namespace tnt;

__device__ uint64_t mix(uint64_t z) {  // splitmix64
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
__device__ double at_exp(uint64_t mant, int ex) { return __longlong_as_double((long long)((uint64_t)(1023 + ex) << 52 | (mant >> 12))); }
// max of non-negative doubles by their bits
__device__ void put(unsigned long long* w, double v) { atomicMax(w, (unsigned long long)__double_as_longlong(v)); }

__global__ void k_check(unsigned long long* worst, unsigned* bad, int n) {
  double mr = 0, mq = 0;
  unsigned b = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint64_t m = mix((uint64_t)i);
    if (i % 4 == 0) m = (uint64_t)(i / 4 % 4096) << 12;    // next to 1
    if (i % 4 == 1) m = ~((uint64_t)(i / 4 % 4096) << 12);  // next to 2
    // reciprocal
    const double d = at_exp(m, 0), q = rcp_newton(d);
    mr = fmax(mr, fabs(fma(-d, q, 1.0)));
    const int k = (int)(mix(m + i) % (922 + 1022 + 1)) - 1022;
    b += rcp_newton(at_exp(m, k)) != ldexp(q, -k);
    b += rcp_newton(-at_exp(m, k)) != -ldexp(q, -k);
    // reciprocal root: odd and even exponents
    const double s = at_exp(m, i / 8 % 2), y = rsqrt_newton(s), p = y * y, pe = fma(y, y, -p);
    mq = fmax(mq, 0.5 * fabs(fma(-s, p, 1.0) - s * pe));
    const int h = (int)(mix(m - i) % 1022) - 511;
    b += rsqrt_newton(at_exp(m, i / 8 % 2 + 2 * h)) != ldexp(y, -h);
  }
  put(worst, mr);
  put(worst + 1, mq);
  if (b) atomicAdd(bad, b);
}

int main() {
  unsigned long long* w;
  unsigned* bad;
  if (cudaMallocManaged(&w, 16) != cudaSuccess || cudaMallocManaged(&bad, 4) != cudaSuccess) return 2;
  w[0] = w[1] = 0;
  *bad = 0;
  k_check<<<304, 256>>>(w, bad, 1 << 26);
  if (cudaDeviceSynchronize() != cudaSuccess) return 2;
  double r[2];
  for (int i = 0; i < 2; ++i) r[i] = double_of_bits(w[i]) * 9007199254740992.0;  // in 2^-53
  std::printf("rcp %.5f rsqrt %.5f of 2^-53, scaled copies that differ %u\n", r[0], r[1], *bad);
  return r[0] <= 1.001 && r[1] <= 1.501 && *bad == 0 ? 0 : 1;
}
