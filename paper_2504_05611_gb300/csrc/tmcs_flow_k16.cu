// Decoupled event-signature kernels, tiles of 16 chunks (tmcs_flow.cuh).
#include "tmcs_flow.cuh"

namespace tmcs {
TMCS_FLOW_UNIT(16)
}  // namespace tmcs
