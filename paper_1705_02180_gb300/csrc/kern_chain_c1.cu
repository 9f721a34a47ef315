// Chain kernels: one CTA per replica (up to 1024 threads) or frame.
#include "kern_chain.cuh"

namespace scps {
SCPS_RESIDENT_LAUNCHERS(, 1, false)
SCPS_EVAL_LAUNCHERS(, 1)
}  // namespace scps
