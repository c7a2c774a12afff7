// Decoupled event-signature kernels, tiles of 4 chunks (tmcs_flow.cuh).
#include "tmcs_flow.cuh"

namespace tmcs {
TMCS_FLOW_UNIT(4)
}  // namespace tmcs
