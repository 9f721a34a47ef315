// Chain kernels: two CTAs per replica or frame.
#include "kern_chain.cuh"

namespace scps {
SCPS_RESIDENT_LAUNCHERS(, 2, true)
SCPS_EVAL_LAUNCHERS(, 2)
}  // namespace scps
