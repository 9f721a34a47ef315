// Chain kernels: four CTAs per replica or frame.
#include "kern_chain.cuh"

namespace scps {
SCPS_RESIDENT_LAUNCHERS(, 4, true)
SCPS_EVAL_LAUNCHERS(, 4)
SCPS_MAX_CLUSTERS(, 4)
}  // namespace scps
