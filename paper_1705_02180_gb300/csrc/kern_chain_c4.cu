// Chain kernels on clusters of 4 CTAs per replica or frame.
#include "kern_chain.cuh"

namespace scps {
SCPS_CHAIN_LAUNCHERS(, 4)
}  // namespace scps
