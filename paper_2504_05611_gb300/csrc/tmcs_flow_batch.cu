// Decoupled event-signature kernel over many circuits (tmcs_flow.cuh).
#include "tmcs_flow.cuh"

namespace tmcs {

__global__ void __launch_bounds__(TMCS_FLOW_MAX_THREADS, 1) flow_batch_kernel(const __grid_constant__ FlowBatchArgs B) {
    extern __shared__ __align__(128) uint64_t smem[];
    __shared__ FlowCtl C;
    uint32_t lo = 0, hi = B.n_jobs - 1u;
    while (lo < hi) {
        const uint32_t mid = (lo + hi + 1u) / 2u;
        if (B.cta_begin[mid] <= blockIdx.x) lo = mid;
        else hi = mid - 1u;
    }
    const FlowArgs &A = B.jobs[lo];
    const uint32_t bx = blockIdx.x - B.cta_begin[lo], gx = B.cta_begin[lo + 1u] - B.cta_begin[lo];
    switch (B.variant[lo]) {
    case 0: flow_cta<kFlowBatchK, false, false, 3>(A, smem, C, bx, gx); break;
    case 1: flow_cta<kFlowBatchK, true, false, 3>(A, smem, C, bx, gx); break;
    case 2: flow_cta<kFlowBatchK, false, true, 2>(A, smem, C, bx, gx); break;
    case 3: flow_cta<kFlowBatchK, true, true, 2>(A, smem, C, bx, gx); break;
    case 4: flow_cta<kFlowBatchK, false, true, 3>(A, smem, C, bx, gx); break;
    default: flow_cta<kFlowBatchK, true, true, 3>(A, smem, C, bx, gx); break;
    }
}

cudaError_t flow_batch_launch(const FlowBatchArgs &b, int threads, size_t smem, cudaStream_t st) {
    cudaError_t e = cudaFuncSetAttribute(flow_batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(flow_batch_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             int(cudaSharedmemCarveoutMaxShared));
    if (e != cudaSuccess) return e;
    flow_batch_kernel<<<b.cta_begin[b.n_jobs], threads, smem, st>>>(b);
    return cudaGetLastError();
}

}  // namespace tmcs
