// Chain kernels: eight CTAs per replica or frame.
#include "kern_chain.cuh"

namespace scps {
SCPS_RESIDENT_LAUNCHERS(, 8, true)
SCPS_EVAL_LAUNCHERS(, 8)
SCPS_MAX_CLUSTERS(, 8)
}  // namespace scps
