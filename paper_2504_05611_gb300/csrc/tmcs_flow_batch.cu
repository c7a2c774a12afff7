// Decoupled event-signature kernels over many circuits (tmcs_flow.cuh). The
// general kernel has windows of three calls, the fast one of two and three.
#include "tmcs_flow.cuh"

namespace tmcs {

template <bool WIDE>
static cudaError_t batch_w(const FlowBatchArgs &b, bool fast, int window, int threads, size_t smem, cudaStream_t st) {
    if (!fast) return flow_batch_go<WIDE, false, 3>(b, threads, smem, st);
    return window <= 2 ? flow_batch_go<WIDE, true, 2>(b, threads, smem, st)
                       : flow_batch_go<WIDE, true, 3>(b, threads, smem, st);
}

cudaError_t flow_batch_launch(const FlowBatchArgs &b, bool wide, bool fast, int window, int threads, size_t smem,
                              cudaStream_t st) {
    return wide ? batch_w<true>(b, fast, window, threads, smem, st)
                : batch_w<false>(b, fast, window, threads, smem, st);
}

}  // namespace tmcs
