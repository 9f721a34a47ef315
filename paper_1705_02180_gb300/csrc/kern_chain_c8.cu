// Chain kernels on clusters of 8 CTAs per replica or frame.
#include "kern_chain.cuh"

namespace scps {
SCPS_CHAIN_LAUNCHERS(, 8)
}  // namespace scps
