// Decoupled event-signature kernels, tiles of 8 chunks (tmcs_flow.cuh).
#include "tmcs_flow.cuh"

namespace tmcs {
TMCS_FLOW_UNIT(8)
}  // namespace tmcs
