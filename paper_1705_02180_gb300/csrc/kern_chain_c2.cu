// Chain kernels on clusters of 2 CTAs per replica or frame.
#include "kern_chain.cuh"

namespace scps {
SCPS_CHAIN_LAUNCHERS(, 2)
}  // namespace scps
