// Advance-kernel instantiations whose warps work in pairs (256-thread blocks).
#include "lpm_advance.cuh"

namespace lpm {
LPM_ADVANCE_PAIR_TU(256)
}  // namespace lpm
