// How a Krylov step's vectors are dealt to the CTAs of the one-launch Gram-Schmidt step
// (kernels_f64.cu), and where it applies.  Plain host code, checked by tests/gs_split_host.cu.
#pragma once
#include <cstddef>
#include <cstdint>

namespace tnt {

constexpr size_t GS_SMEM = 204 * 1024;
// Above this both forms are bound by the FP64 pipe.  FP64 solves of this size, fused (then with
// two passes over all of V) / separate launches: n = 2^12 9.7 / 27 ms, 2^16 28 / 50, 2^18 60 / 80,
// 2^20 232 / 239.
constexpr int64_t GS_MAX_N = 1 << 20;

// elements of w per CTA: as many CTAs as SMs, down to 64 elements each
inline int64_t gs_slice(int64_t n, int nsm) {
  const int64_t s = (n + nsm - 1) / nsm;
  return s < 64 ? 64 : s;
}
// a CTA keeps its slice of w in shared memory: with 80 SMs visible that holds a little less
// than GS_MAX_N entries
inline bool gs_fits(int64_t n, int nsm) { return n <= GS_MAX_N && 16 * (size_t)gs_slice(n, nsm) <= GS_SMEM; }

}  // namespace tnt
