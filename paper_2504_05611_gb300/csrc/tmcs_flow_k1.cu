// Decoupled event-signature kernels, tiles of 1 chunk (tmcs_flow.cuh).
#include "tmcs_flow.cuh"

namespace tmcs {
TMCS_FLOW_UNIT(1)
}  // namespace tmcs
