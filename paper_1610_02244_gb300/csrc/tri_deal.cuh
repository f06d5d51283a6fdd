// How the blocks of one SVD are dealt to the SMs for the reduction with rows in shared memory
// (k_tridiag_group, heig.cu).  Plain host code, checked by tests/tri_deal_host.cu for any
// number of SMs.
#pragma once
#include <cstddef>
#include <cstdint>
#include <vector>

namespace tnt {

constexpr int64_t TRI_ROWS_NMAX = 1216;  // the kernel's vectors: three entries per thread of 512, with room
constexpr int TRI_RMAX = 128;            // rows per CTA
constexpr int TRI_MAXB = 48;             // blocks of one launch

// whether a group of q CTAs with `smem` bytes each holds the rows of an m x m block and its
// three vectors (four in a group of one CTA)
inline bool tri_fits(int64_t m, int64_t q, size_t smem) {
  const int64_t rows = (m + q - 1) / q;
  return rows <= TRI_RMAX && (size_t)(rows + 3 + (q == 1)) * (size_t)m * 16 <= smem;
}
// Whether nsm SMs hold the block at all.  152 SMs hold eight rows each of 1216; 148 would need
// nine, which with the vectors pass the shared memory of an SM above 1184 rows.
inline bool tri_holds(int64_t m, int nsm, size_t smem) {
  return m <= TRI_ROWS_NMAX && (tri_fits(m, 1, smem) || tri_fits(m, m < nsm ? m : nsm, smem));
}

// CTAs of each block's group (in the order of `n`, descending) for one launch on nsm SMs of
// smem bytes: the shortest common time by the model
//   t(n, nb) = n t_col + (2 n^3 / nb + 4 n^2) / f,
// 12 FP64 operations per trailing entry of a CTA's rows and 16 per entry of its vectors at two
// per SM and clock, and a column's latency t_col (scalars, loads, barrier: 4 us in a group
// of one CTA, 5 us and 0.01 us per CTA with a barrier).  Returns how many of the blocks fit the launch.
inline int tri_deal(const std::vector<int64_t>& n, int nsm, size_t smem, std::vector<int>* nb) {
  auto time = [](double m, double q) { return m * (q > 1 ? 5.0 + 0.01 * q : 4.0) + (2.0 * m * m * m / q + 4.0 * m * m) / 2070.0; };
  std::vector<int> lo;
  int used = 0;
  for (int64_t m : n) {  // the least group that holds each block
    int q = 1;
    while (q < m && !tri_fits(m, q, smem)) ++q;
    if (!tri_fits(m, q, smem) || used + q > nsm || (int)lo.size() == TRI_MAXB) break;
    lo.push_back(q);
    used += q;
  }
  const int cnt = (int)lo.size();
  // more CTAs to the block that takes longest, as long as that shortens it
  std::vector<int> q = lo;
  while (cnt > 0) {
    int w = 0;
    for (int i = 1; i < cnt; ++i)
      if (time((double)n[(size_t)i], q[(size_t)i]) > time((double)n[(size_t)w], q[(size_t)w])) w = i;
    const double m = (double)n[(size_t)w], now = time(m, q[(size_t)w]);
    // the next size worth having: a second CTA brings the barrier's cost with it
    int next = q[(size_t)w] + 1;
    while (next - q[(size_t)w] <= nsm - used && next < (int)m && time(m, next) >= now) ++next;
    if (next - q[(size_t)w] > nsm - used || next > (int)m || time(m, next) >= now) break;
    used += next - q[(size_t)w];
    q[(size_t)w] = next;
  }
  *nb = q;
  return cnt;
}

}  // namespace tnt
