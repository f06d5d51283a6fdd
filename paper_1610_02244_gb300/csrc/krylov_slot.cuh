// What k_tridiag_lowest writes to pinned memory for one Krylov step, and how the host reads it.
// The device's status word travels with the numbers: a CTA whose barrier wait expires leaves
// without its slice of the next basis vector, while the others, CTA 0 among them, may still
// pass the barrier and leave a finite beta.
#pragma once
#include <cmath>

namespace tnt {

struct KrylovSlot {
  double E, ylast, beta, status;
};
enum SlotState { SLOT_OK = 0, SLOT_TIMEOUT, SLOT_NAN };
inline SlotState slot_state(const KrylovSlot& s) {
  if (s.status != 0.0) return SLOT_TIMEOUT;
  return std::isfinite(s.E) && std::isfinite(s.beta) ? SLOT_OK : SLOT_NAN;
}

}  // namespace tnt
