// Host check of csrc/tri_deal.cuh for any number of visible SMs: a block is either held by a group
// (and then dealt at once) or takes the other route; groups stay within the SMs, the rows and
// the shared memory; every list of held blocks is worked off.
#include <algorithm>
#include <cstdio>

#include "tri_deal.cuh"

int main() {
  using namespace tnt;
  const size_t smem = 227 * 1024 - 5000;
  int bad = 0;
  long held = 0, refused = 0;
  for (int nsm : {1, 2, 7, 20, 66, 76, 132, 144, 148, 151, 152, 160}) {
    for (int64_t m = 1; m <= 1400; ++m) {
      std::vector<int> q;
      const bool h = tri_holds(m, nsm, smem);
      (h ? held : refused)++;
      const int cnt = m <= TRI_ROWS_NMAX ? tri_deal({m}, nsm, smem, &q) : 0;
      bad += (cnt == 1) != h;
      if (cnt == 1) bad += q[0] < 1 || q[0] > nsm || q[0] > m || !tri_fits(m, q[0], smem);
      if (m > TRI_ROWS_NMAX) bad += h;
    }
    // a mixed list, the largest first
    std::vector<int64_t> n;
    for (int64_t m : {1216, 1200, 1184, 900, 700, 500, 300, 300, 200, 130, 120, 64, 33, 8, 1, 1})
      if (tri_holds(m, nsm, smem)) n.push_back(m);
    for (int i = 0; i < 60; ++i) n.push_back(1);
    for (size_t i = 0; i < n.size();) {
      std::vector<int> q;
      const int cnt = tri_deal({n.begin() + i, n.end()}, nsm, smem, &q);
      int used = 0;
      for (int k = 0; k < cnt; ++k) {
        used += q[(size_t)k];
        bad += !tri_fits(n[i + (size_t)k], q[(size_t)k], smem);
      }
      bad += used > nsm || cnt > TRI_MAXB;
      if (cnt < 1) {
        ++bad;
        break;
      }
      i += (size_t)cnt;
    }
  }
  // the whole range on 152 SMs; part of it on 148
  bad += !tri_holds(1216, 152, smem) || tri_holds(1217, 152, smem) || tri_holds(1200, 148, smem) || !tri_holds(1184, 148, smem);
  std::printf("held %ld refused %ld mismatches %d\n", held, refused, bad);
  return bad ? 1 : 0;
}
