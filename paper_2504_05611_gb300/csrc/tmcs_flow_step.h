#pragma once
// Completion of a step in the decoupled kernel (tmcs_flow.cuh): how the
// walkers report a step's batches and put-aside blocks, and what the appliers
// wait for. Written over the accesses to the step's slot (S), so that the
// same code runs in the kernel and, interleaved in every order, on the CPU
// (tests/flow_step_model.cpp).
//
// S has: add_batch(), counts one batch as walked (acquire and release) and
// returns the count before; add_unit(), counts one finished block (release);
// done(), the counts, batches | units << 16 (acquire); left(), the streams
// put aside (final once every batch is counted).
#include <cstdint>

#ifdef __CUDACC__
#define TMCS_STEP_FN __host__ __device__ __forceinline__
#else
#define TMCS_STEP_FN inline
#endif

namespace tmcs {

// A walker's report of one walked batch of a step with nb batches and room
// for lcap put-aside streams (whole blocks of 32). full() finishes the blocks
// that this batch filled and counts each; part(block, n) finishes the n
// streams of the last, partial block without counting it.
//
// The walker of the step's last batch reads left() and counts one closing
// unit after it, whether or not a partial block is left. Until then the step
// is not complete, so its slot and region are not reused: without the unit a
// step with no partial block would be complete with the batch count alone,
// and the read of left() could meet the count of the step kFlowSlots later.
template <class S, class Full, class Part>
TMCS_STEP_FN void flow_batch_walked(S &s, uint32_t nb, uint32_t lcap, Full &&full, Part &&part) {
    const uint32_t before = s.add_batch();
    full();
    if ((before & 0xFFFFu) != nb - 1u) return;
    const uint32_t left = s.left();
    const uint32_t n = left < lcap ? left : lcap;
    if (n & 31u) part(n >> 5, n & 31u);
    s.add_unit();
}

// Whether a step of nb batches is complete: all batches walked, every full
// block of put-aside streams finished, and the closing unit counted.
template <class S>
TMCS_STEP_FN bool flow_step_complete(S &s, uint32_t nb, uint32_t lcap) {
    const uint32_t d = s.done();
    if ((d & 0xFFFFu) != nb) return false;
    if (nb == 0u) return true;
    const uint32_t left = s.left();
    return (d >> 16) == (left < lcap ? left : lcap) / 32u + 1u;
}

}  // namespace tmcs
