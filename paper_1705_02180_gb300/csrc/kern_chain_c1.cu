// Chain kernels on clusters of 1 CTA per replica or frame.
#include "kern_chain.cuh"

namespace scps {
SCPS_CHAIN_LAUNCHERS(, 1)
}  // namespace scps
