// Host check of csrc/krylov_slot.cuh: an expired wait is reported whatever the numbers say.
#include <cstdio>

#include "krylov_slot.cuh"

int main() {
  using namespace tnt;
  int bad = 0;
  const double vals[] = {0.0, -1.5, 1e300, INFINITY, -INFINITY, NAN};
  for (double E : vals)
    for (double b : vals) {
      const bool fin = std::isfinite(E) && std::isfinite(b);
      bad += slot_state(KrylovSlot{E, 0.5, b, 0.0}) != (fin ? SLOT_OK : SLOT_NAN);
      for (double st : {1.0, 2.0, 3.0}) bad += slot_state(KrylovSlot{E, 0.5, b, st}) != SLOT_TIMEOUT;
    }
  std::printf("mismatches %d\n", bad);
  return bad ? 1 : 0;
}
