// Decoupled event-signature kernels, tiles of 2 chunks (tmcs_flow.cuh).
#include "tmcs_flow.cuh"

namespace tmcs {
TMCS_FLOW_UNIT(2)
}  // namespace tmcs
