#pragma once
// Decoupled event-signature sampler (sm_103a): the walk of the noise streams
// and the application of their events to the detector words run in
// different warps, joined by a shared-memory event arena instead of CTA
// barriers.
//
// What it computes is what sig_kernel computes (Methods "Simulation":
// detector and observable flips as XORs of the output lists of the sampled
// noise events, each event drawn from the Philox4x32-10 streams of the
// sampling specification), with the same schedule: items (64-unit noise
// segments) in steps whose detectors lie in a ring window above the step's
// flush point. The difference is the execution:
//
//  * Walker warps take batches of 32 streams (tile, step, 32 / K items x K
//    chunks) in CTA order from one shared counter, across step and tile
//    boundaries, and append every event that flips something as one 32-bit
//    word (event slot, chunk, lane) to their step's region of a circular
//    arena.
//  * Applier warps take steps in order: once every stream of step Q has
//    finished, they apply its events to the ring (shared-memory atomic XORs
//    of the ring rows in the event's slot), write the detectors the step
//    finalises to HBM, clear them, and free the step's arena region.
//
// A step's region has a capacity fixed at launch from the expected number
// of its events (mean + 6 sigma + 64) and of its streams that a batch puts
// aside. A walker may start a batch of step Q only when Q's region no longer
// overlaps an unapplied step's; an event beyond its region's capacity is held
// by its lane, which waits until Q is the step being applied and then XORs
// the event into the ring itself before its batch counts as walked. The ring
// is therefore only ever touched for the step being applied, so it needs one
// window of detectors, while the arena keeps several steps of walking in
// flight. All waits are bounded (kWaitNs); on expiry the kernel sets bit 0
// of the status word and every warp leaves.
//
// Measured (one GB300, 2070 MHz; before = one lane per stream with refills,
// 8-byte event slots per Pauli index): d=29 non-local CNOT, p = 1e-3, 2e6
// shots (12.39 GB of output): 11.2 ms before, 9.4 ms now (1.32 TB/s); the
// same at p = 1e-4: 6.6, 4.9 (2.5 TB/s); d=11, 1e7 shots: 3.28, 2.61; BB144
// teleport, 3e6: 3.02, 1.97. What bounds it now is the appliers' chain: a
// step of d=29 costs them 6.6 k cycles of application, 4.2 k of flush and 1.1 k
// of waiting.
#include <cuda.h>  // CUtensorMap (encoded through the runtime's driver entry point)
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "tmcs_device.cuh"
#include "tmcs_flow_step.h"
#include "tmcs_internal.h"

namespace tmcs {

constexpr uint32_t kFlowSlots = 16;       // steps in flight (done / count slots)
// events an applier lane loads at once (build-time tuning value)
#ifndef TMCS_FLOW_APPLY_BATCH
#define TMCS_FLOW_APPLY_BATCH 4
#endif
constexpr uint32_t kFlowApplyBatch = TMCS_FLOW_APPLY_BATCH;
constexpr uint32_t kFlowBlocks = 32;      // blocks of 32 put-aside streams a step has at most
constexpr uint32_t kFlowMinArena = 1024;  // smallest useful arena (entries)
constexpr uint32_t kFlowMaxArena = 65536;
struct FlowArgs {
    CUtensorMap tmap;           // det as a [n_det][ld] uint64 tensor (tensor-store flush), when tma_rows > 0
    const NoiseDesc *noise;
    const uint32_t *tables;
    const uint4 *item_desc;     // walker descriptors, two uint4 per item (see SigSchedule::item_desc)
    const uint4 *steps;         // item_begin, item_end, flush_lo, flush_hi
    const float *step_events;   // per step: expected live events, unfinished streams by window (SigSchedule)
    const uint32_t *rows;       // ring rows of every compact event slot (see SigSchedule::rows)
    uint32_t n_steps, window_mask, n_obs;
    uint32_t arena;             // arena entries
    uint32_t test_cap;          // testing: capacity of every step's region (0: from step_events)
    uint32_t pc1;               // the program has PAULI_CHANNEL_1 noise
    uint32_t near;              // every gap table allows the one-read count (kNearInv)
    uint32_t smem_tables;       // gap tables staged in shared memory (count), 0: read from global
    uint32_t walkers;           // walker warps; the CTA's other warps apply
    uint32_t key0, key1, first_chunk;
    PhiloxKeys keys;            // round keys of rounds 2..10
    uint32_t vec_out;           // det 16-byte aligned and n_cols even: 16-byte output stores
    uint64_t n_cols, last_mask, n_tiles;
    uint64_t ld;                // words between output rows (the call's column count; a launch may cover a slice)
    uint32_t tma_rows;          // detector rows per tensor-store box of the flush (0: plain stores)
    uint64_t col_base;          // column of this launch's column 0 in the tensor map (sliced launches)
    uint64_t *det;
    uint64_t *obs;
    uint32_t *status;
};

// Step positions in the arena's sequence are kept modulo 2^32: only
// differences (less than the arena size plus one step's region) are used.
struct FlowCtl {
    uint32_t next;                 // batches handed out (CTA sequence; a launch keeps it below 2^31)
    uint32_t u_applied;            // arena position of the first unapplied step
    uint32_t applied;              // steps applied (CTA sequence)
    uint32_t abort;                // a bounded wait expired
    uint32_t app_stop;             // appliers leave (written by applier thread 0 before a barrier)
    // of step Q, in slot Q mod kFlowSlots:
    uint32_t done[kFlowSlots];     // walked batches | units << 16 (finished blocks of put-aside streams, closing unit)
    uint32_t cnt[kFlowSlots];      // arena entries reserved by its events
    uint32_t left[kFlowSlots];     // streams put aside
    uint32_t blk[kFlowSlots][kFlowBlocks / 4];  // entries written per block of 32 (a byte each)
};

static_assert(sizeof(FlowCtl) <= 1024, "the launch leaves 1 KB for static shared variables");

// Shared-memory regions (same order and sizes as flow_fixed_bytes): ring and
// observable rows, step table (batches up to and including the step, region
// capacity for events, for put-aside streams, region offset; then the tile's
// total), gap tables, arena.
struct FlowSmem {
    uint64_t *ring;
    uint32_t *bend, *scap, *slcap, *soff;
    uint32_t *stab;
    uint32_t *arena;
};

__host__ __device__ inline size_t flow_ring_bytes(uint32_t W, uint32_t n_obs, int K) {
    // detectors, observables and the spare row
    return ((size_t(W) + n_obs + 1) * size_t(K) * 8 + 15) & ~size_t(15);
}
__host__ __device__ inline size_t flow_step_bytes(uint32_t n_steps) {
    return ((4 * size_t(n_steps) + 1) * 4 + 15) & ~size_t(15);
}

__device__ __forceinline__ FlowSmem flow_layout(uint64_t *smem, const FlowArgs &A, int K) {
    FlowSmem S;
    unsigned char *b = reinterpret_cast<unsigned char *>(smem);
    S.ring = smem;
    b += flow_ring_bytes(A.window_mask + 1u, A.n_obs, K);
    S.bend = reinterpret_cast<uint32_t *>(b);
    S.scap = S.bend + A.n_steps;
    S.slcap = S.scap + A.n_steps;
    S.soff = S.slcap + A.n_steps;
    b += flow_step_bytes(A.n_steps);
    S.stab = reinterpret_cast<uint32_t *>(b);
    b += size_t(A.smem_tables) * kTableWords * 4;
    S.arena = reinterpret_cast<uint32_t *>(b);
    return S;
}

template <int K>
struct FlowLog {
    static constexpr uint32_t v = K == 1 ? 0 : K == 2 ? 1 : K == 4 ? 2 : K == 8 ? 3 : 4;
};

// One compact event slot as loaded, two rows per word (see
// SigSchedule::rows); the last word is two rows or the link to the next chunk
// of a long list.
template <bool WIDE>
struct FlowSlot;
template <>
struct FlowSlot<false> {
    uint32_t x, last;
    __device__ __forceinline__ static FlowSlot load(const uint32_t *rows, uint32_t slot) {
        const uint2 v = __ldg(reinterpret_cast<const uint2 *>(rows) + slot);
        return {v.x, v.y};
    }
};
template <>
struct FlowSlot<true> {
    uint32_t x, y, z, last;
    __device__ __forceinline__ static FlowSlot load(const uint32_t *rows, uint32_t slot) {
        const uint4 v = __ldg(reinterpret_cast<const uint4 *>(rows) + slot);
        return {v.x, v.y, v.z, v.w};
    }
};

// XORs the rows of one loaded chunk into the ring for event word wv = event
// slot << (6 + log2 K) | chunk << 6 | lane. Unused entries name the spare
// row, so a pair is applied without tests; a word of two of them ends the
// list.
template <int K, bool WIDE>
__device__ __forceinline__ void flow_put(const FlowArgs &A, uint64_t *ring, uint32_t wv, const FlowSlot<WIDE> &v) {
    // 32-bit word of the row that holds the event's lane: 2 chunk + lane / 32
    uint32_t *const base = reinterpret_cast<uint32_t *>(ring) + ((wv >> 5) & (2u * uint32_t(K) - 1u));
    const uint32_t bit = 1u << (wv & 31u);
    const uint32_t spare = (A.window_mask + 1u + A.n_obs) * 0x10001u;
    auto pair = [&](uint32_t w) {
        atomicXor(base + (w & 0xFFFFu) * (2u * uint32_t(K)), bit);
        atomicXor(base + (w >> 16) * (2u * uint32_t(K)), bit);
    };
    pair(v.x);
    if constexpr (WIDE) {
        if (v.y == spare) return;
        pair(v.y);
        if (v.z == spare) return;
        pair(v.z);
    }
    if (v.last != spare && !(v.last & kRowOverflow)) pair(v.last);
}

// One event from its slot on, chunk by chunk.
template <int K, bool WIDE>
__device__ __forceinline__ void flow_put_all(const FlowArgs &A, uint64_t *ring, uint32_t wv, FlowSlot<WIDE> v) {
    for (;;) {
        flow_put<K, WIDE>(A, ring, wv, v);
        if (!(v.last & kRowOverflow)) return;
        v = FlowSlot<WIDE>::load(A.rows, v.last & ~kRowOverflow);
    }
}

// Waits until done() holds, polled by lane 0 for the whole warp; bounded
// (kWaitNs). False for every lane when the wait expired, here (status bit
// set) or in another warp.
template <class Done>
__device__ __forceinline__ bool flow_warp_wait(FlowCtl &C, uint32_t *status, uint32_t lane, Done &&done) {
    int ok = 1;
    if (lane == 0 && !done()) {
        const uint64_t t0 = globaltimer_ns();
        while (!done()) {
            if (ld_shared_volatile(&C.abort)) {
                ok = 0;
                break;
            }
            if (globaltimer_ns() - t0 > kWaitNs) {
                C.abort = 1u;
                atomicOr(status, 1u);
                ok = 0;
                break;
            }
            __nanosleep(64);
        }
    }
    // the shuffle carries the decision, the warp barrier lane 0's acquire
    ok = __shfl_sync(0xFFFFFFFFu, ok, 0);
    __syncwarp();
    return ok != 0;
}

// Accesses to a step's slot by a whole walker warp (lane 0 does the atomics).
struct FlowStepWarp {
    FlowCtl &C;
    uint32_t slot, lane;
    __device__ __forceinline__ uint32_t add_batch() {
        uint32_t old = 0;
        __syncwarp();
        if (lane == 0) old = atom_add_acq_rel_shared(&C.done[slot], 1u);
        return __shfl_sync(0xFFFFFFFFu, old, 0);
    }
    __device__ __forceinline__ void add_unit() {
        __syncwarp();
        if (lane == 0) red_release_add_shared(&C.done[slot], 0x10000u);
    }
    __device__ __forceinline__ uint32_t left() { return ld_acquire_shared(&C.left[slot]); }
};
// The same by one applier thread.
struct FlowStepThread {
    FlowCtl &C;
    uint32_t slot;
    __device__ __forceinline__ uint32_t done() { return ld_acquire_shared(&C.done[slot]); }
    __device__ __forceinline__ uint32_t left() { return ld_shared_volatile(&C.left[slot]); }
};

// Walker warps.
//
// A batch is 32 streams of one step: 32 / K consecutive items x the tile's K
// chunks, one per lane (lane = item x K + chunk), so everything but the
// stream itself is uniform over the warp: the step, its arena region, the
// gate, the completion. Batches are handed out in CTA order (tile, step,
// batch) from one shared counter. A batch runs a first window of W Philox
// calls (two draws each; W from the items' expected draws, the same for the
// 32 streams, which are sorted by that) as straight-line code. The streams
// that need more draws (a few of the 32) are put aside, one word each, in
// the tail of the step's arena region; the warp whose streams fill a block
// of 32 there finishes that block, the warp that walks the step's last batch
// the rest. Running on in place with the few lanes that are not done would
// cost a call per batch at a fifth of the lanes.
//
// What bounds it: instruction issue (the integer pipe and the 64-bit
// products of Philox, four issue cycles each, above all). One lane per
// stream with refills after every window (the layout this replaced) spent
// 310 of its 830 warp-instructions per iteration on per-lane bookkeeping:
// refill, gate, grouping lanes by step, completion.
// FAST: gap tables in shared memory, one table read per gap count, no
// PAULI_CHANNEL_1 noise (a program without ebit decoherence, every p above
// 2.1e-5); the other cases share the general kernel (tables through L1),
// which counts gaps with one read in batches whose tables all allow it. Two
// kernels instead of run-time branches: the walkers' code is about the size of
// the instruction caches, and every branch not taken sits between the ones
// that are (stalls without an instruction were 1.6 of 12.7 cycles per issue).
// W: Philox calls of every stream's first window. One length per launch (the
// best for the program's items together): kernels with all four lengths and a
// choice per batch measured 320 against 310 ns per chunk on d=29, 2.78 against
// 2.70 ms on BB144 teleport, for the same reason.
template <int K, bool FAST, bool WIDE, int W>
struct FlowWalker {
    static constexpr bool SMT = FAST;
    static constexpr uint32_t LK = FlowLog<K>::v;
    static constexpr uint32_t IPB = 32u / uint32_t(K);  // items per batch
    static constexpr uint32_t S_EV = 6u + LK;           // event words: slot << S_EV | chunk << 6 | lane
    static constexpr uint32_t CB = WIDE ? 4u : 2u;      // bits of a class

    const FlowArgs &A;
    const FlowSmem &S;
    FlowCtl &C;
    const uint32_t *tabs;
    uint32_t lane, lt;
    uint32_t bx, gx;  // the CTA among those of its job, their number
    // the step being walked: sequence number, first item, item end, batches,
    // region (position in the arena, capacity for events and for put-aside
    // streams), tile's first chunk, valid chunks
    uint32_t Q = 0xFFFFFFFFu, item0 = 0, item_end = 0, nb = 0, upos = 0, cap = 0, lcap = 0, chunk0 = 0, nv = 0;

    struct Stream {
        PhiloxStream ps;
        uint32_t evb, kpm, npm, tab1, kind, desc;
        uint64_t lut;  // classes << S_EV - CB shifted right by a Pauli index's bits (CB per index)
        int n_trials;
        float inv, c32;
    };

    // Decodes the lane's stream: item (index in the schedule), chunk k of
    // the tile. Event words are slot << S_EV | chunk << 6 | lane with slot =
    // slot0 + (pos >> 6) classes + class - 1, formed as evb + (pos >> 6) kpm
    // + pos + class << S_EV (modulo 2^32).
    __device__ __forceinline__ Stream open(uint32_t item, uint32_t k, bool valid) const {
        const uint4 d0 = __ldg(A.item_desc + 2 * item), d1 = __ldg(A.item_desc + 2 * item + 1);
        Stream s;
        s.kind = d1.x & 7u;
        s.npm = ((d1.x >> 3) & 15u) * CB;
        s.kpm = (((d1.x >> 7) & 15u) << S_EV) - 64u;
        s.tab1 = (d1.x >> 19) * kTableWords - 1u;
        s.desc = d1.z;
        // four-row layout: 30 bits, kept S_EV bits up so that the shift by a
        // Pauli index leaves its class in place in the event word
        s.lut = WIDE ? uint64_t(d1.y) | (uint64_t(d1.z) << 32) : uint64_t(d1.y) << S_EV;
        s.inv = __uint_as_float(d1.w);
        s.c32 = -32.0f * s.inv;  // exact (a power-of-two scaling)
        // Philox round 1 from the descriptor's product of the op index
        // (counter words: call, chunk, op, segment)
        s.ps.a0 = d0.x ^ (chunk0 + k) ^ A.key0;
        s.ps.a1 = d0.y;
        s.ps.a3 = d0.z ^ A.key1;
        s.evb = ((d0.w - 1u) << S_EV) + (k << 6);
        // lanes past the step's items and chunks past the call's end: no trials
        s.n_trials = valid ? 64 * int(((d1.x >> 11) & 63u) + 1u) : 0;
        return s;
    }

    // Waits until the step's arena region is free (`gate`: signed difference
    // modulo 2^32) and the step is within the slots in flight. False when a
    // bounded wait expired, here or elsewhere.
    __device__ __forceinline__ bool wait_gate(uint32_t gate) const {
        return flow_warp_wait(C, A.status, lane, [&]() {
            // acquire: the appliers' last reads of the region and their
            // reset of the step's counters precede our writes
            return int32_t(ld_acquire_shared(&C.u_applied) - gate) >= 0 &&
                   Q - ld_acquire_shared(&C.applied) < kFlowSlots;
        });
    }

    // Event of a lane whose step's region is full: the lane waits until the
    // step is the one being applied (the ring then holds its window) and
    // XORs the event into the ring itself. Every earlier step can finish
    // without this warp: it has reported all its batches of those. When the
    // bounded wait expires the event is dropped, the status bit set, and the
    // warp leaves at its next gate.
    __device__ __noinline__ static void put_late(const FlowArgs &A, uint64_t *ring, FlowCtl &C, uint32_t Q, uint32_t wv) {
        const uint64_t t0 = globaltimer_ns();
        while (ld_acquire_shared(&C.applied) != Q) {
            if (ld_shared_volatile(&C.abort)) return;
            if (globaltimer_ns() - t0 > kWaitNs) {
                C.abort = 1u;
                atomicOr(A.status, 1u);
                return;
            }
            __nanosleep(64);
        }
        flow_put_all<K, WIDE>(A, ring, wv, FlowSlot<WIDE>::load(A.rows, wv >> S_EV));
    }

    // Stores the lane's events of a window (those with live[d]) in the step's
    // arena region, next to one another. Every lane reserves its entries with
    // its own shared atomic: the warp's same-address adds cost the memory
    // pipe a cycle a lane, ballots and population counts for one add per warp
    // cost the integer pipes more (d=29 workload: 263 k against 244 k
    // warp-instructions a chunk, 388 against 345 ns). One counter per step:
    // regions in 2 / 4 / 8 parts with a counter each, so that fewer lanes
    // share an address, measured 304 / 320 / 330 against 293 ns (the appliers'
    // lanes then read events of more items at once).
    template <int NE>
    __device__ __forceinline__ void emit(const uint32_t (&ev)[NE], const bool (&live)[NE]) const {
        uint32_t n = 0;
#pragma unroll
        for (int d = 0; d < NE; d++) n += live[d] ? 1u : 0u;
        uint32_t idx = 0;
        if (n) idx = atomicAdd(&C.cnt[Q & (kFlowSlots - 1u)], n);
        uint32_t a = upos + idx;
        if (a >= A.arena) a -= A.arena;
        if (a + uint32_t(NE) <= A.arena && idx + uint32_t(NE) <= cap) {
            uint32_t *at = S.arena + a;
#pragma unroll
            for (int d = 0; d < NE; d++) {
                if (live[d]) *at = ev[d];
                at += live[d] ? 1 : 0;
            }
        } else {
            // near the arena's end or the region's
#pragma unroll
            for (int d = 0; d < NE; d++)
                if (live[d]) {
                    if (idx < cap) S.arena[a] = ev[d];
                    else put_late(A, S.ring, C, Q, ev[d]);
                    idx++;
                    a = a + 1u < A.arena ? a + 1u : 0u;
                }
        }
    }

    // V Philox calls from call `call` on, 2V draws: positions in draw order
    // (increasing), the events before the end of the segment stored. NEAR:
    // one table read per gap count (gap_count_near_at's derivation), the
    // estimate rounded by adding 1.5 x 2^23 so that the table index is the
    // sum's low bits.
    template <int V, bool NEAR>
    __device__ __forceinline__ void window(const Stream &s, uint32_t call, int &pos, bool walk) const {
        constexpr int NE = 2 * V;
        uint32_t wp[NE];
        int pd[NE];
#pragma unroll
        for (int c = 0; c < V; c++) {
            const uint4 w = philox_call(s.ps, call + uint32_t(c), A.keys);
            if constexpr (NEAR) {
                pd[2 * c] = gap_count_magic<SMT>(tabs, s.tab1, s.inv, s.c32, w.x);
                pd[2 * c + 1] = gap_count_magic<SMT>(tabs, s.tab1, s.inv, s.c32, w.z);
            } else {
                pd[2 * c] = gap_count_est<SMT>(tabs + (s.tab1 + 1u), s.inv, s.c32, w.x);
                pd[2 * c + 1] = gap_count_est<SMT>(tabs + (s.tab1 + 1u), s.inv, s.c32, w.z);
            }
            wp[2 * c] = w.y;
            wp[2 * c + 1] = w.w;
        }
        const int n_trials = walk ? s.n_trials : 0;
        uint32_t ev[NE];
        bool live[NE];
        auto words = [&](auto pc1) {
            uint32_t t1 = 0, t2 = 0;
            if constexpr (decltype(pc1)::value)
                if (s.kind == N_PC1) {
                    t1 = __ldg(&A.noise[s.desc].t1);
                    t2 = __ldg(&A.noise[s.desc].t2);
                }
#pragma unroll
            for (int d = 0; d < NE; d++) {
                pos += 1 + pd[d];
                // CB x (Pauli index - 1): floor(CB n w / 2^32) without its
                // low bits, as floor(n w / 2^32) = floor(floor(CB n w / 2^32) / CB)
                uint32_t kb = __umulhi(wp[d], s.npm) & ~(CB - 1u);
                if constexpr (decltype(pc1)::value)
                    if (s.kind == N_PC1) kb = wp[d] < t1 ? 0u : wp[d] < t2 ? 2u * CB : CB;
                const uint32_t pu = uint32_t(pos);
                uint32_t cls;  // class << S_EV
                if constexpr (WIDE) cls = (uint32_t(s.lut >> kb) & 15u) << S_EV;
                else cls = uint32_t(s.lut >> kb) & (3u << S_EV);
                ev[d] = (pu >> 6) * s.kpm + (s.evb + pu + cls);
                live[d] = pos < n_trials && cls != 0u;
            }
        };
        if constexpr (FAST) {
            words(std::false_type{});
        } else {
            if (A.pc1) words(std::true_type{});
            else words(std::false_type{});
        }
        emit<NE>(ev, live);
    }

    // Runs the lanes with `walk` to the end of their streams, a call at a
    // time. near: every lane's table allows the one-read count.
    __device__ __forceinline__ void finish(const Stream &s, uint32_t call, int pos, bool walk, bool near) const {
        while (__any_sync(0xFFFFFFFFu, walk)) {
            if (FAST || near) window<1, true>(s, call, pos, walk);
            else window<1, false>(s, call, pos, walk);
            call++;
            walk = walk && pos < s.n_trials;
        }
    }

    // Puts the lanes' unfinished streams (mask um, not 0) aside. Returns the
    // blocks of 32 that are complete with them (bits 0 and 1: the block
    // whose number is in the bits above and the next one; 0: none). Entry:
    // position | lane << 12 | batch within the step << 17. Only batches that
    // had a first window put streams aside, so all tables here are near.
    __device__ __forceinline__ uint32_t put_aside(const Stream &s, uint32_t um, uint32_t b, int pos) const {
        const uint32_t slot = Q & (kFlowSlots - 1u), n = uint32_t(__popc(um));
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(&C.left[slot], n);
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        const bool mine = (um >> lane) & 1u;
        const uint32_t idx = base + uint32_t(__popc(um & lt));
        if (mine && idx < lcap) {
            const uint32_t a = upos + cap + idx;
            S.arena[a >= A.arena ? a - A.arena : a] = uint32_t(pos) | (lane << 12) | (b << 17);
        }
        __syncwarp();
        // count the entries written per block (they touch two blocks at
        // most: lanes 0 and 1); the warp that completes a block's count has
        // acquired every entry of it and finishes it, without a wait. Both
        // blocks can become complete here: the second one's other entries
        // may have been written first.
        bool full = false;
        const uint32_t lo = min(base, lcap), hi = min(base + n, lcap);
        if (lane < 2) {
            const uint32_t bk = (lo >> 5) + lane, f = max(lo, bk << 5), e = min(hi, (bk + 1u) << 5);
            if (f < e) {
                const uint32_t sh = 8u * (bk & 3u);
                const uint32_t old = atom_add_acq_rel_shared(&C.blk[slot][bk >> 2], (e - f) << sh);
                full = ((old >> sh) & 255u) + (e - f) == 32u;
            }
        }
        const uint32_t fm = __ballot_sync(0xFFFFFFFFu, full);
        // the region's tail is full: finish in place
        if (base + n > lcap) finish(s, uint32_t(W), pos, mine && idx >= lcap, true);
        return fm ? (lo >> 5) << 2 | fm : 0u;
    }

    // Finishes n streams put aside in block `blk` (the caller counts the block).
    __device__ __forceinline__ void finish_block(uint32_t blk, uint32_t n) const {
        __syncwarp();  // the entries, acquired by one lane
        const bool have = lane < n;
        // lanes without an entry take the step's first stream, in the general
        // kernel the last entry's (its table is a near one)
        const uint32_t a = upos + cap + 32u * blk + (FAST ? lane : min(lane, n - 1u));
        const uint32_t e = !FAST || have ? S.arena[a >= A.arena ? a - A.arena : a] : 0u;
        const uint32_t sl = (e >> 12) & 31u;
        const uint32_t item = item0 + (e >> 17) * IPB + (sl >> LK);
        const Stream s = open(item, sl & uint32_t(K - 1), have);
        finish(s, uint32_t(W), int(e & 0xFFFu), have, true);
    }

    __device__ void run(uint32_t nt, uint32_t nv_last) {
        const uint32_t n_steps = A.n_steps;
        const uint32_t bpt = S.bend[n_steps - 1u];  // batches per tile
        const uint32_t total = nt * bpt;
        const uint32_t c_tile = S.soff[n_steps];
        uint32_t T = 0, q = 0, tb = 0;  // the tile and step of the batch last taken, the tile's first batch
        uint32_t b0 = 0;                // the step's first batch in the tile
        for (;;) {
            uint32_t g = 0;
            if (lane == 0) g = atomicAdd(&C.next, 1u);
            g = __shfl_sync(0xFFFFFFFFu, g, 0);
            if (g >= total) return;
            while (g - tb >= bpt) {
                tb += bpt;
                T++;
                q = 0;
            }
            while (g - tb >= S.bend[q]) q++;
            if (Q != T * n_steps + q) {
                Q = T * n_steps + q;
                const uint4 st = __ldg(A.steps + q);
                item0 = st.x;
                item_end = st.y;
                b0 = q ? S.bend[q - 1u] : 0u;
                nb = S.bend[q] - b0;
                cap = S.scap[q];
                lcap = S.slcap[q];
                const uint32_t U = T * c_tile + S.soff[q];  // modulo 2^32
                upos = uint32_t((uint64_t(T) * c_tile + S.soff[q]) % A.arena);
                chunk0 = A.first_chunk + (bx + T * gx) * uint32_t(K);
                nv = T == nt - 1u ? nv_last : uint32_t(K);
                if (!wait_gate(U + cap + lcap - A.arena)) return;
            }
            const uint32_t b = g - tb - b0;
            const uint32_t k = lane & uint32_t(K - 1);
            const uint32_t it = item0 + b * IPB + (lane >> LK);
            const Stream s = open(min(it, item_end - 1u), k, it < item_end && k < nv);
            int pos = -1;
            // The one-read count is a choice per batch: a table of p below
            // 2.1e-5 in one noise op must not take the first window from
            // every other stream (as one choice per launch did: d=11
            // decoherence workload with aged-ebit ops of p = 1.5e-5, 1e6 shots,
            // 433 us against 290; without the small p 291 us).
            const bool near = FAST || A.near || __all_sync(0xFFFFFFFFu, fabsf(s.inv) < kNearInv);
            if (near) window<W, true>(s, 0u, pos, true);
            const bool unfinished = pos < s.n_trials && s.n_trials > 0;
            const uint32_t um = __ballot_sync(0xFFFFFFFFu, unfinished);
            uint32_t full = 0;
            if (um != 0) {
                // finish in place when most lanes go on, when there was no
                // first window (a table needs the two-read count), and when
                // the batch number does not fit an entry
                if (!near) finish(s, 0u, pos, unfinished, false);
                else if (__popc(um) > 24 || b >= (1u << 15)) finish(s, uint32_t(W), pos, unfinished, true);
                else full = put_aside(s, um, b, pos);
            }
            // the batch is walked (release: its events and entries are in the
            // arena or the ring)
            FlowStepWarp step{C, Q & (kFlowSlots - 1u), lane};
            flow_batch_walked(
                step, nb, lcap,
                [&]() {
                    if (full & 1u) {
                        finish_block(full >> 2, 32u);
                        step.add_unit();
                    }
                    if (full & 2u) {
                        finish_block((full >> 2) + 1u, 32u);
                        step.add_unit();
                    }
                },
                [&](uint32_t blk, uint32_t n) { finish_block(blk, n); });
        }
    }
};

__device__ __forceinline__ void flow_bar(uint32_t nthreads) {
    asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

__device__ __forceinline__ void fence_proxy_async_shared() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, int x, int y, const void *src) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(shared_addr(src))
                 : "memory");
}
__device__ __forceinline__ void tma_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void tma_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void tma_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Rows [d0, d1) of one contiguous stretch of the ring: plain head rows
// [d0, dh) up to the first 128-byte aligned ring row, whole boxes [dh, db),
// plain tail rows [db, d1).
struct FlushSeg {
    uint32_t d0, dh, db, d1;
};

template <int K>
__device__ __forceinline__ FlushSeg flush_seg(uint32_t d, uint32_t e, uint32_t mask, uint32_t R) {
    constexpr uint32_t AL = K >= 16 ? 1u : 16u / uint32_t(K);  // ring rows per 128 bytes
    FlushSeg g;
    g.d0 = d;
    g.d1 = e;
    g.dh = min(e, d + (AL - (d & mask) % AL) % AL);
    g.db = g.dh + (e - g.dh) / R * R;
    return g;
}

template <int K>
__device__ __forceinline__ void flush_plain_rows(const FlowArgs &A, const FlowSmem &S, const FlushSeg &g,
                                                 uint64_t col0, uint32_t nv, uint32_t at, uint32_t nthr) {
    const uint32_t nh = g.dh - g.d0, nt = g.d1 - g.db;
    for (uint32_t i = at; i < (nh + nt) * uint32_t(K); i += nthr) {
        const uint32_t row = i / uint32_t(K), k = i % uint32_t(K);
        const uint32_t d = row < nh ? g.d0 + row : g.db + (row - nh);
        uint64_t *r = S.ring + size_t(d & A.window_mask) * K + k;
        const uint64_t v = *r;
        *r = 0ull;
        if (k < nv) __stcs(reinterpret_cast<unsigned long long *>(A.det + uint64_t(d) * A.ld + col0 + k), v);
    }
}

template <int K>
__device__ __forceinline__ void flush_clear_boxes(const FlowArgs &A, const FlowSmem &S, const FlushSeg &g,
                                                  uint32_t at, uint32_t nthr) {
    ulonglong2 *base = reinterpret_cast<ulonglong2 *>(S.ring + size_t(g.dh & A.window_mask) * K);
    const uint32_t nw = (g.db - g.dh) * uint32_t(K) / 2u;
    for (uint32_t i = at; i < nw; i += nthr) base[i] = make_ulonglong2(0ull, 0ull);
}

// Flush of detectors [z, w) (w - z at most the ring's rows) with tensor
// stores: the rows of each stretch of the ring (at most two: the ring wraps)
// go out as boxes of tma_rows rows x K chunk words issued by the first
// applier warp, each starting at a 128-byte aligned ring row; the few rows
// before the first aligned row and after the last whole box are written with
// plain stores. Every row is cleared: the boxes' rows once the tensor stores
// have read them. The call's last column (in the call's last tile) gets its
// pad bits masked in the ring first. Every applier has fenced its ring
// writes for the async proxy before the barrier that precedes this call.
// Ends with the boxes' rows cleared; the caller's barrier follows.
template <int K>
__device__ __forceinline__ void flow_flush_tma(const FlowArgs &A, const FlowSmem &S, uint32_t z, uint32_t w,
                                               uint64_t col0, uint32_t nv, uint32_t at, uint32_t nthr) {
    const uint32_t mask = A.window_mask, R = A.tma_rows;
    if (col0 + uint64_t(K) > A.n_cols - 1) {  // this tile holds the call's last column
        const uint32_t kl = uint32_t(A.n_cols - 1 - col0);
        for (uint32_t i = at; i < w - z; i += nthr) S.ring[size_t((z + i) & mask) * K + kl] &= A.last_mask;
        fence_proxy_async_shared();
        flow_bar(nthr);
    }
    const uint32_t split = min(w, z + (mask + 1u - (z & mask)));  // first row past the ring's end
    const FlushSeg g0 = flush_seg<K>(z, split, mask, R), g1 = flush_seg<K>(split, w, mask, R);
    const uint32_t n0 = (g0.db - g0.dh) / R, nbox = n0 + (g1.db - g1.dh) / R;
    const bool issuer = at < 32u;
    if (issuer) {
        const int x = int(A.col_base + col0);
        for (uint32_t b = at; b < nbox; b += 32u) {
            const uint32_t d = b < n0 ? g0.dh + b * R : g1.dh + (b - n0) * R;
            tma_store_2d(&A.tmap, x, int(d), S.ring + size_t(d & mask) * K);
        }
        tma_commit();
    }
    flush_plain_rows<K>(A, S, g0, col0, nv, at, nthr);
    flush_plain_rows<K>(A, S, g1, col0, nv, at, nthr);
    if (issuer) tma_wait_read();
    flow_bar(nthr);
    flush_clear_boxes<K>(A, S, g0, at, nthr);
    flush_clear_boxes<K>(A, S, g1, at, nthr);
}

// Applier warps: steps in CTA order.
template <int K, bool WIDE>
__device__ __forceinline__ void flow_apply(const FlowArgs &A, const FlowSmem &S, FlowCtl &C, uint32_t nt,
                                           uint32_t nv_last, uint32_t bx, uint32_t gx) {
    constexpr uint32_t LK = FlowLog<K>::v, S_EV = 6u + LK;
    const uint32_t nthr = blockDim.x - 32u * A.walkers;
    const uint32_t at = threadIdx.x - 32u * A.walkers;
    const uint32_t mask = A.window_mask;
    const uint32_t obs_row = A.window_mask + 1u;
    const uint32_t *const arena = S.arena;
    // tensor-store flush: needs the ring 128-byte aligned in shared memory
    // and boxes of a whole number of 128-byte ring stretches (each box then
    // starts aligned)
    const bool tma = (K % 2 == 0) && A.tma_rows != 0 && (A.tma_rows * uint32_t(K)) % 16u == 0 &&
                     (shared_addr(S.ring) & 127u) == 0;
    uint32_t U = 0;   // arena position of step Q, modulo 2^32
    uint32_t up = 0;  // the same modulo the arena size
    for (uint32_t T = 0; T < nt; T++) {
        const uint64_t tile = uint64_t(bx) + uint64_t(T) * gx;
        const uint64_t col0 = tile * uint64_t(K);
        const uint32_t nv = T == nt - 1u ? nv_last : uint32_t(K);
        for (uint32_t q = 0; q < A.n_steps; q++) {
            const uint32_t Q = T * A.n_steps + q;
            const uint4 st = __ldg(A.steps + q);
            const uint32_t need = S.bend[q] - (q ? S.bend[q - 1u] : 0u);
            const uint32_t slot = Q & (kFlowSlots - 1u);
            // thread 0 waits for the step's streams and decides for all
            // appliers whether they go on (one value read after the barrier,
            // so every applier thread leaves or none does)
            if (at == 0) {
                FlowStepThread step{C, slot};
                auto complete = [&]() { return flow_step_complete(step, need, S.slcap[q]); };
                uint32_t stop = ld_shared_volatile(&C.abort);
                if (!stop && !complete()) {
                    const uint64_t t0 = globaltimer_ns();
                    while (!complete()) {
                        if (ld_shared_volatile(&C.abort)) {
                            stop = 1u;
                            break;
                        }
                        if (globaltimer_ns() - t0 > kWaitNs) {
                            C.abort = 1u;
                            atomicOr(A.status, 1u);
                            stop = 1u;
                            break;
                        }
                        __nanosleep(32);
                    }
                }
                C.app_stop = stop;
            }
            flow_bar(nthr);
            if (C.app_stop) {
                if (tma && at < 32u) tma_wait_all();
                return;
            }
            __threadfence_block();  // the walkers' events precede the reads below
            const uint32_t cap = S.scap[q];
            const uint32_t n = min(ld_shared_volatile(&C.cnt[slot]), cap);
            // Batches of kFlowApplyBatch events per thread: their slot loads
            // overlap, then their rows are applied, then the next chunks of
            // those with long lists are loaded together, and so on. (Each
            // event's list followed to its end before the next event cost a
            // dependent L2 read per event: with two rows per slot 2 % of the
            // events of a surface code had one, so half of all warp-wide
            // events did.)
            const uint32_t per = nthr * kFlowApplyBatch;
            auto entry = [&](uint32_t i) {
                const uint32_t a = up + i;
                return arena[a >= A.arena ? a - A.arena : a];
            };
            for (uint32_t e = at; e < n; e += per) {
                uint32_t wv[kFlowApplyBatch];
                FlowSlot<WIDE> v[kFlowApplyBatch];
#pragma unroll
                for (uint32_t j = 0; j < kFlowApplyBatch; j++) wv[j] = entry(min(e + j * nthr, n - 1u));
#pragma unroll
                for (uint32_t j = 0; j < kFlowApplyBatch; j++) v[j] = FlowSlot<WIDE>::load(A.rows, wv[j] >> S_EV);
                uint32_t go = 0;  // bit j: event j has a chunk to apply
#pragma unroll
                for (uint32_t j = 0; j < kFlowApplyBatch; j++) go |= e + j * nthr < n ? 1u << j : 0u;
                for (;;) {
                    uint32_t more = 0;
#pragma unroll
                    for (uint32_t j = 0; j < kFlowApplyBatch; j++)
                        if ((go >> j) & 1u) {
                            flow_put<K, WIDE>(A, S.ring, wv[j], v[j]);
                            more |= (v[j].last >> 31) << j;
                        }
                    if (!more) break;
                    go = more;
#pragma unroll
                    for (uint32_t j = 0; j < kFlowApplyBatch; j++)
                        if ((go >> j) & 1u) v[j] = FlowSlot<WIDE>::load(A.rows, v[j].last & ~kRowOverflow);
                }
            }
            if (tma) fence_proxy_async_shared();  // ring writes before the tensor stores read them
            flow_bar(nthr);
            // every applier has read the step's arena entries (barrier): the
            // region is free for the walkers of later steps while the
            // appliers flush (release: those reads precede the hand-off)
            U += cap + S.slcap[q];
            up += cap + S.slcap[q];
            if (up >= A.arena) up -= A.arena;
            if (at == 0) st_release_shared(&C.u_applied, U);
            // detectors [flush_lo, flush_hi) are final: write and clear them
            const uint32_t nd = st.w - st.z;
            bool vec_done = false;
            if constexpr (K % 2 == 0) {
                if (tma) {
                    vec_done = true;
                    flow_flush_tma<K>(A, S, st.z, st.w, col0, nv, at, nthr);
                } else if (A.vec_out) {
                    vec_done = true;
                    constexpr uint32_t H = uint32_t(K) / 2u;
                    for (uint32_t i = at; i < nd * H; i += nthr) {
                        const uint32_t d = st.z + i / H, k = 2u * (i % H);
                        ulonglong2 *r = reinterpret_cast<ulonglong2 *>(S.ring + size_t(d & mask) * K + k);
                        ulonglong2 v = *r;
                        *r = make_ulonglong2(0ull, 0ull);
                        if (k >= nv) continue;
                        const uint64_t col = col0 + k;
                        if (col == A.n_cols - 1) v.x &= A.last_mask;
                        if (col + 1 == A.n_cols - 1) v.y &= A.last_mask;
                        unsigned long long *out =
                            reinterpret_cast<unsigned long long *>(A.det + uint64_t(d) * A.ld + col);
                        if (k + 1 < nv) __stcs(reinterpret_cast<ulonglong2 *>(out), v);
                        else __stcs(out, v.x);
                    }
                }
            }
            if (!vec_done) {
                for (uint32_t i = at; i < nd * uint32_t(K); i += nthr) {
                    const uint32_t d = st.z + i / uint32_t(K), k = i % uint32_t(K);
                    uint64_t *r = S.ring + size_t(d & mask) * K + k;
                    uint64_t v = *r;
                    *r = 0ull;
                    if (k >= nv) continue;
                    const uint64_t col = col0 + k;
                    if (col == A.n_cols - 1) v &= A.last_mask;
                    __stcs(reinterpret_cast<unsigned long long *>(A.det + uint64_t(d) * A.ld + col), v);
                }
            }
            if (q == A.n_steps - 1u) {
                uint64_t *ob = S.ring + size_t(obs_row) * K;
                for (uint32_t i = at; i < A.n_obs * uint32_t(K); i += nthr) {
                    const uint32_t o = i / uint32_t(K), k = i % uint32_t(K);
                    uint64_t v = ob[i];
                    ob[i] = 0ull;
                    if (k >= nv) continue;
                    const uint64_t col = col0 + k;
                    if (col == A.n_cols - 1) v &= A.last_mask;
                    A.obs[uint64_t(o) * A.ld + col] = v;
                }
            }
            flow_bar(nthr);
            if (at == 0) {
                C.done[slot] = 0u;
                C.cnt[slot] = 0u;
                C.left[slot] = 0u;
#pragma unroll
                for (uint32_t i = 0; i < kFlowBlocks / 4; i++) C.blk[slot][i] = 0u;
                // release: every applier's ring writes of this step (ordered
                // before by the barrier) and the counter resets precede the
                // hand-off of the ring window and the step's slots
                st_release_shared(&C.applied, Q + 1u);
            }
        }
    }
    if (tma && at < 32u) tma_wait_all();  // the tensor stores have written the outputs
}

// CTA size the kernel is compiled for (its register budget follows from it)
#ifndef TMCS_FLOW_MAX_THREADS
#define TMCS_FLOW_MAX_THREADS 1024
#endif

// One CTA (number bx of gx) of a job: tiles bx, bx + gx, ...
template <int K, bool WIDE, bool FAST, int W>
__device__ __forceinline__ void flow_cta(const FlowArgs &A, uint64_t *smem, FlowCtl &C, uint32_t bx, uint32_t gx) {
    if (uint64_t(bx) >= A.n_tiles) return;
    const FlowSmem S = flow_layout(smem, A, K);
    const uint32_t tid = threadIdx.x, T_ = blockDim.x;
    const uint32_t rows = A.window_mask + 1u;
    for (uint32_t i = tid; i < (rows + A.n_obs) * uint32_t(K); i += T_) S.ring[i] = 0ull;
    for (uint32_t i = tid; i < A.smem_tables * kTableWords; i += T_) S.stab[i] = __ldg(A.tables + i);
    // batches per step (prefix sum below) and region capacities: mean + 6 sigma + 64 of the step's events over K
    // chunks (Poisson-like counts), at most the arena; steps without items
    // hold none (flow_region, tmcs_flow.cu, has the same formulas)
    for (uint32_t i = tid; i < A.n_steps; i += T_) {
        const uint4 st = __ldg(A.steps + i);
        const float mu = __ldg(A.step_events + 5 * i) * float(K), ml = __ldg(A.step_events + 5 * i + W) * float(K);
        uint32_t cap = A.test_cap ? A.test_cap : uint32_t(ceilf(mu + 6.0f * sqrtf(mu) + 64.0f));
        // put-aside streams: whole blocks, at most a quarter of the arena
        uint32_t lcap = min((uint32_t(ceilf(ml + 6.0f * sqrtf(ml))) + 63u) & ~31u, (A.arena / 4u) & ~31u);
        lcap = st.y > st.x ? min(lcap, 32u * kFlowBlocks) : 0u;
        cap = st.y > st.x ? min(cap, A.arena - lcap) : 0u;
        S.bend[i] = (st.y - st.x + 32u / uint32_t(K) - 1u) / (32u / uint32_t(K));
        S.scap[i] = cap;
        S.slcap[i] = lcap;
    }
    if (tid < kFlowSlots) {
        C.done[tid] = 0u;
        C.cnt[tid] = 0u;
        C.left[tid] = 0u;
        for (uint32_t i = 0; i < kFlowBlocks / 4; i++) C.blk[tid][i] = 0u;
    }
    if (tid == 0) {
        C.next = 0u;
        C.u_applied = 0u;
        C.applied = 0u;
        C.abort = 0u;
        C.app_stop = 0u;
    }
    __syncthreads();
    // region offsets: exclusive prefix sum of the capacities (warp 0);
    // batches: inclusive prefix sum (warp 1)
    if (tid < 64) {
        const bool bat = tid >= 32;
        const uint32_t l = tid & 31u;
        const uint32_t per = (A.n_steps + 31u) / 32u, lo = min(A.n_steps, l * per), hi = min(A.n_steps, lo + per);
        uint32_t sum = 0;
        for (uint32_t i = lo; i < hi; i++) sum += bat ? S.bend[i] : S.scap[i] + S.slcap[i];
        uint32_t incl = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (int(l) >= o) incl += v;
        }
        uint32_t run = incl - sum;
        for (uint32_t i = lo; i < hi; i++) {
            if (bat) {
                run += S.bend[i];
                S.bend[i] = run;
            } else {
                S.soff[i] = run;
                run += S.scap[i] + S.slcap[i];
            }
        }
        if (!bat && l == 31) S.soff[A.n_steps] = incl;
    }
    const uint32_t nt = uint32_t((A.n_tiles - bx + gx - 1) / gx);
    const uint64_t last = uint64_t(bx) + uint64_t(nt - 1) * gx;
    const uint64_t rem = A.n_cols - last * K;
    const uint32_t nv_last = rem < uint64_t(K) ? uint32_t(rem) : uint32_t(K);
    __syncthreads();
    if ((tid >> 5) >= A.walkers) {
        flow_apply<K, WIDE>(A, S, C, nt, nv_last, bx, gx);
    } else {
        const uint32_t lane = tid & 31u;
        FlowWalker<K, FAST, WIDE, W> w{A, S, C, FAST ? S.stab : A.tables, lane, (1u << lane) - 1u, bx, gx};
        w.run(nt, nv_last);
    }
}

template <int K, bool WIDE, bool FAST, int W>
__global__ void __launch_bounds__(TMCS_FLOW_MAX_THREADS, 1) flow_kernel(const __grid_constant__ FlowArgs A) {
    extern __shared__ __align__(128) uint64_t smem[];
    __shared__ FlowCtl C;
    flow_cta<K, WIDE, FAST, W>(A, smem, C, blockIdx.x, gridDim.x);
}

// Many small circuits in one launch: every CTA works on one job, and a job
// has as many CTAs as its share of the work (the host's choice), so the jobs
// run side by side and none waits for a launch of its own. The job table is
// a kernel parameter, so a graph can hold the launch. Tiles of four chunks:
// the jobs are those that do not fill the GPU alone.
//
// A job's variant (slot layout, fast or general walker, first window) is a
// branch per CTA, so jobs of all kinds share the launch. One launch per
// variant let the longest step chain of each kind follow the others': four
// small circuits of four kinds 43.5 us against 31.7, a batch of 16
// distance-5 to 9 and BB18 circuits 100 us against 80.
constexpr int kFlowBatchK = 4;
constexpr uint32_t kFlowBatchJobs = 64;
struct FlowBatchArgs {
    FlowArgs jobs[kFlowBatchJobs];
    uint32_t cta_begin[kFlowBatchJobs + 1];  // first CTA of each job; [n_jobs] = all
    uint32_t n_jobs;
    uint8_t variant[kFlowBatchJobs];         // flow_batch_variant
};
static_assert(sizeof(FlowBatchArgs) <= 32000, "the job table exceeds the kernel parameter limit");

// The general kernel has windows of three calls here, the fast one of two and
// three.
inline uint8_t flow_batch_variant(bool wide, bool fast, int window) {
    return uint8_t((wide ? 1 : 0) + (!fast ? 0 : window <= 2 ? 2 : 4));
}

cudaError_t flow_batch_launch(const FlowBatchArgs &b, int threads, size_t smem, cudaStream_t st);

// Launch of one kernel variant: a persistent grid of the CTAs that are
// resident at once, never more than there are tiles.
template <int K, bool WIDE, bool FAST, int W>
cudaError_t flow_go(const FlowArgs &a, const FlowShape &s, int sms, cudaStream_t st) {
    auto kern = flow_kernel<K, WIDE, FAST, W>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(s.smem));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, int(cudaSharedmemCarveoutMaxShared));
    if (e != cudaSuccess) return e;
    // a CTA of more than 512 threads at this register budget leaves no room
    // for a second one; smaller ones are asked for
    int per_sm = 1;
    if (s.threads <= 512) {
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, s.threads, s.smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorInvalidConfiguration;
    }
    const uint64_t grid = std::max<uint64_t>(1, std::min<uint64_t>(a.n_tiles, uint64_t(sms) * uint64_t(per_sm)));
    kern<<<unsigned(grid), s.threads, s.smem, st>>>(a);
    return cudaGetLastError();
}

// The variants of one tile size (each tile size is a translation unit, so
// that they compile in parallel). The general kernel has windows of one and
// three calls.
template <int K, bool WIDE>
cudaError_t flow_go_w(const FlowArgs &a, const FlowShape &s, int sms, cudaStream_t st) {
    if (!s.fast) return s.window <= 1 ? flow_go<K, WIDE, false, 1>(a, s, sms, st) : flow_go<K, WIDE, false, 3>(a, s, sms, st);
    switch (s.window) {
    case 1: return flow_go<K, WIDE, true, 1>(a, s, sms, st);
    case 2: return flow_go<K, WIDE, true, 2>(a, s, sms, st);
    case 3: return flow_go<K, WIDE, true, 3>(a, s, sms, st);
    default: return flow_go<K, WIDE, true, 4>(a, s, sms, st);
    }
}

#define TMCS_FLOW_UNIT(K)                                                                                  \
    cudaError_t flow_go_##K(const FlowArgs &a, const FlowShape &s, bool wide, int sms, cudaStream_t st) {   \
        return wide ? flow_go_w<K, true>(a, s, sms, st) : flow_go_w<K, false>(a, s, sms, st);               \
    }

cudaError_t flow_go_1(const FlowArgs &a, const FlowShape &s, bool wide, int sms, cudaStream_t st);
cudaError_t flow_go_2(const FlowArgs &a, const FlowShape &s, bool wide, int sms, cudaStream_t st);
cudaError_t flow_go_4(const FlowArgs &a, const FlowShape &s, bool wide, int sms, cudaStream_t st);
cudaError_t flow_go_8(const FlowArgs &a, const FlowShape &s, bool wide, int sms, cudaStream_t st);
cudaError_t flow_go_16(const FlowArgs &a, const FlowShape &s, bool wide, int sms, cudaStream_t st);

}  // namespace tmcs
