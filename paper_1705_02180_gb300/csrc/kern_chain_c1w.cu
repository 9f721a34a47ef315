// Chain kernels: one CTA per replica, with an SM to itself.
#include "kern_chain.cuh"

namespace scps {
SCPS_RESIDENT_LAUNCHERS(, 1, true)
}  // namespace scps
