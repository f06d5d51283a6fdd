// Host check of csrc/gs_split.cuh for any number of visible SMs: where the one-launch step
// applies its slices cover the vector, one per SM at most, and fit the shared memory.
#include <cstdio>

#include "gs_split.cuh"

int main() {
  using namespace tnt;
  int bad = 0;
  for (int nsm : {1, 2, 20, 66, 79, 80, 81, 132, 148, 152, 160}) {
    for (int64_t n = 1; n <= GS_MAX_N + 3; n += 1 + n / 97) {
      const int64_t S = gs_slice(n, nsm), grid = (n + S - 1) / S;
      const bool room = 16 * (size_t)S <= GS_SMEM;
      bad += S < 64 || grid < 1 || grid > nsm || grid * S < n;
      bad += gs_fits(n, nsm) != (room && n <= GS_MAX_N);
    }
  }
  bad += !gs_fits(GS_MAX_N, 152) || gs_fits(GS_MAX_N + 1, 152) || gs_fits(GS_MAX_N, 80) || !gs_fits(1 << 19, 80);
  std::printf("mismatches %d\n", bad);
  return bad ? 1 : 0;
}
