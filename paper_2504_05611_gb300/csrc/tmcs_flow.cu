// Host side of the decoupled event-signature sampler (kernels: tmcs_flow.cuh;
// one translation unit per tile size, tmcs_flow_k*.cu): launch shape, tensor
// map of the output, launches over column slices.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "tmcs_flow.cuh"

namespace tmcs {

static int env_int_flow(const char *name, int dflt) {
    const char *v = std::getenv(name);
    return (v && *v) ? std::atoi(v) : dflt;
}

static size_t flow_fixed_bytes(const SigProgram &G, int sched, uint32_t n_obs, int K) {
    const SigSchedule &S = G.sched[sched];
    return flow_ring_bytes(S.window, n_obs, K) + flow_step_bytes(uint32_t(S.steps.size()));
}

// Arena region of a step with mu expected events and ml expected put-aside
// streams (the kernel's formulas, flow_cta; in one function for both, the
// kernel's set-up compiled to code that made it 0.6 % slower).
static double flow_region(float mu, float ml, uint32_t arena) {
    const double blocks = double((uint64_t(std::ceil(ml + 6.0f * std::sqrt(ml))) + 63u) & ~uint64_t(31));
    return std::ceil(mu + 6.0 * std::sqrt(mu) + 64.0) +
           std::min({blocks, double((arena / 4u) & ~31u), double(32u * kFlowBlocks)});
}

bool flow_shape(const tmcs_circuit *c, int sched, int K, int threads, int appliers, size_t budget, FlowShape *out) {
    const SigProgram &G = c->sig;
    if (!G.ok || sched < 0 || size_t(sched) >= G.sched.size()) return false;
    const SigSchedule &S = G.sched[sched];
    if (S.lag || S.rows.empty() || S.steps.empty() || S.steps.size() > kFlowMaxSteps ||
        S.step_events.size() != 5 * S.steps.size())
        return false;
    if (K != 1 && K != 2 && K != 4 && K != 8 && K != 16) return false;
    if (threads < 64 || threads > TMCS_FLOW_MAX_THREADS || threads % 32 || appliers < 1 || appliers >= threads / 32)
        return false;
    // event words: slot << (6 + log2 K) | chunk << 6 | lane must fit 32 bits
    if (G.n_compact_slots * 64u * uint64_t(K) >= (uint64_t(1) << 32)) return false;
    // batches of a step are counted in 16 bits
    for (const SigStep &t : S.steps)
        if ((t.item_end - t.item_begin) / (32u / uint32_t(K)) >= 65000u) return false;
    const size_t fixed = flow_fixed_bytes(G, sched, uint32_t(c->n_obs), K);
    const size_t tabs = G.tables.size() * 4;
    // what is left of the budget, in entries
    auto arena_for = [&](size_t used) -> uint32_t {
        return used >= budget ? 0u : uint32_t(std::min<size_t>((budget - used) / 4, kFlowMaxArena)) & ~3u;
    };
    FlowShape s;
    s.sched = sched;
    s.K = K;
    s.threads = threads;
    s.appliers = appliers;
    // testing knob: Philox calls of every stream's first window (1 to 4)
    const int wforce = env_int_flow("TMCS_FLOW_WINDOW", 0);
    s.window = (wforce >= 1 && wforce <= 4) ? wforce : int(G.window_calls);
    // gap tables in shared memory when that still leaves an arena of 8192
    // entries, else read through L1
    s.smem_tables = arena_for(fixed + tabs) >= 8192u;
    s.fast = s.smem_tables && G.near && !G.pc1;
    if (!s.fast) s.window = s.window <= 1 ? 1 : 3;  // the general kernel's windows
    s.arena = arena_for(fixed + (s.smem_tables ? tabs : 0));
    const int aforce = env_int_flow("TMCS_FLOW_ARENA", 0);  // tuning/testing knob: arena entries
    if (aforce >= int(kFlowMinArena) && uint32_t(aforce) < s.arena) s.arena = uint32_t(aforce) & ~3u;
    if (s.arena < kFlowMinArena) return false;
    s.smem = fixed + (s.smem_tables ? tabs : 0) + size_t(s.arena) * 4;
    s.regions = double(s.arena) / flow_region(S.max_events * float(K), S.max_left[s.window] * float(K), s.arena);
    // relative time of a tile (see flow_shape_untimed)
    s.cost = double(S.steps.size()) +
             S.sum_events * double(K) / 700.0 * (s.regions < 1.0 ? 2.5 : s.regions < 3.0 ? 1.25 : 1.0);
    *out = s;
    return true;
}

// The ring of least cost: a hand-over per step, and the tile's events, which
// take longer when the arena holds less than three regions (walkers and
// appliers then take turns) and much longer when it holds less than one (the
// events beyond a region wait in the walkers until their step is applied).
// Times of a tile, us, with the steps of a tile and the regions held, for
// rings of 4096 / 2048 / 1024 detectors (d=29: 4096 / 2048), K = 4:
//   d=11, p = 1e-3:  21 (1, 2.5) /  21 (2, 6.5) / 24 (4, 16)
//   d=11, p = 3e-3:  92 (1, 0.9) /  46 (2, 2.3) / 37 (4, 5.8)
//   d=11, p = 1e-2: 289 (1, 0.3) / 306 (2, 0.7) / 130 (4, 1.9)
//   d=21, p = 1e-3:  94 (6, 1.8) /  86 (12, 6.7) / 110 (42, 15)
//   d=29, p = 1e-3: 197 (17, 1.8) / 244 (58, 6.4)
//   BB144 teleport, p = 3e-3: 121 (1, 0.5) / 89 (2, 1.8) / 70 (5, 4.2)
// The weights fit these and the same circuits at K = 1, 2 and 8: 1.2 us a
// step, 1.7 ns an event.
bool flow_shape_untimed(const tmcs_circuit *c, int K, int threads, int appliers, size_t budget, FlowShape *out) {
    bool found = false;
    for (int sched = 0; sched < int(c->sig.sched.size()); sched++) {
        FlowShape s;
        if (!flow_shape(c, sched, K, threads, appliers, budget, &s)) continue;
        if (found && s.cost >= out->cost) continue;
        *out = s;
        found = true;
    }
    return found;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// against the driver library); null if unavailable
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// Tensor map of the call's detector words for the tensor-store flush: a
// [n_det][ld] uint64 tensor, boxes of K chunk words x rows detectors. Needs
// K >= 2 (16-byte box rows), a 16-byte aligned buffer, an even row stride
// and coordinates below 2^31; returns false otherwise.
static bool encode_det_map(CUtensorMap *map, uint64_t *det, uint64_t n_det, uint64_t ld, int K, uint32_t rows) {
    if (K < 2 || !det || reinterpret_cast<uintptr_t>(det) % 16 || ld % 2 || ld >= (uint64_t(1) << 31) ||
        n_det == 0 || n_det >= (uint64_t(1) << 31) || rows == 0 || rows > 256)
        return false;
    const EncodeTiledFn fn = encode_tiled();
    if (!fn) return false;
    const cuuint64_t dim[2] = {ld, n_det};
    const cuuint64_t stride[1] = {ld * 8};
    const cuuint32_t box[2] = {cuuint32_t(K), rows};
    const cuuint32_t estride[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, det, dim, stride, box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
           CUDA_SUCCESS;
}

// What a launch of this shape takes from the program and the call, without
// the columns.
static FlowArgs flow_args(const SigProgram &G, uint32_t n_obs, const DeviceSig *ds, const FlowShape &s,
                          const FlowCall &call) {
    const SigSchedule &S = G.sched[s.sched];
    FlowArgs a{};
    a.noise = ds->noise;
    a.tables = ds->tables;
    a.item_desc = reinterpret_cast<const uint4 *>(ds->item_desc[s.sched]);
    a.steps = reinterpret_cast<const uint4 *>(ds->steps[s.sched]);
    a.step_events = ds->step_events[s.sched];
    a.rows = ds->rows[s.sched];
    a.n_steps = uint32_t(S.steps.size());
    a.window_mask = S.window - 1u;
    a.n_obs = n_obs;
    a.arena = s.arena;
    a.test_cap = uint32_t(std::max(0, env_int_flow("TMCS_TEST_FLOW_CAP", 0)));
    a.pc1 = G.pc1 ? 1u : 0u;
    a.near = G.near ? 1u : 0u;
    a.smem_tables = s.smem_tables ? uint32_t(G.tables.size() / kTableWords) : 0u;
    a.walkers = uint32_t(s.threads / 32 - s.appliers);
    a.key0 = call.key0;
    a.key1 = call.key1;
    a.keys = philox_keys(call.key0, call.key1);
    a.ld = call.ld ? call.ld : call.n_cols;
    a.status = call.status;
    return a;
}

// Columns [c0, c0 + n) of the call.
static void flow_columns(FlowArgs &a, const FlowShape &s, const FlowCall &call, uint64_t c0, uint64_t n) {
    a.first_chunk = call.first_chunk + uint32_t(c0);
    a.n_cols = n;
    a.last_mask = c0 + n == call.n_cols ? call.last_mask : ~uint64_t(0);
    a.n_tiles = (n + uint64_t(s.K) - 1) / uint64_t(s.K);
    a.det = call.det + c0;
    a.col_base = c0;
    a.obs = call.obs ? call.obs + c0 : nullptr;
    a.vec_out = (reinterpret_cast<uintptr_t>(a.det) % 16 == 0 && a.ld % 2 == 0) ? 1u : 0u;
}

static uint64_t batches_per_tile(const SigSchedule &S, int K) {
    const uint64_t ipb = 32u / uint64_t(K);
    uint64_t n = 0;
    for (const SigStep &t : S.steps) n += (t.item_end - t.item_begin + ipb - 1) / ipb;
    return n;
}

int flow_batch_tile() { return kFlowBatchK; }

cudaError_t flow_batch(const std::vector<FlowJob> &jobs, int sms, cudaStream_t st) {
    struct Entry {
        const FlowJob *j;
        FlowArgs a;
        uint8_t variant;
        double tile;  // relative time of a tile
    };
    std::vector<Entry> v;
    v.reserve(jobs.size());
    for (const FlowJob &j : jobs) {
        const SigProgram &G = j.c->sig;
        Entry e{&j, flow_args(G, uint32_t(j.c->n_obs), j.ds, j.shape, j.call), 0, 0.0};
        e.variant = flow_batch_variant(G.wide, j.shape.fast, j.shape.window);
        flow_columns(e.a, j.shape, j.call, 0, j.call.n_cols);
        // batches, events and detectors of a tile, in walker-instruction
        // terms, and the steps' hand-overs (rough weights: they only divide
        // the CTAs among the jobs)
        const SigSchedule &S = G.sched[j.shape.sched];
        double events = 0;
        for (size_t k = 0; k < S.step_events.size(); k += 5) events += double(S.step_events[k]);
        e.tile = 600.0 * double(batches_per_tile(S, kFlowBatchK)) +
                 kFlowBatchK * (2.0 * events + 1.0 * double(G.n_det)) + 2000.0 * double(S.steps.size());
        v.push_back(e);
    }
    for (size_t base = 0; base < v.size(); base += kFlowBatchJobs) {
        const size_t n = std::min<size_t>(kFlowBatchJobs, v.size() - base);
        // CTAs: one each, then one more for the job that would finish
        // last, until every SM has one
        std::vector<uint32_t> ctas(n, 1);
        auto time = [&](size_t i, uint32_t c) {
            const Entry &e = v[base + i];
            return double((e.a.n_tiles + c - 1) / c) * e.tile;
        };
        for (uint32_t used = uint32_t(n); used < uint32_t(sms); used++) {
            size_t worst = 0;
            for (size_t i = 1; i < n; i++)
                if (time(i, ctas[i]) > time(worst, ctas[worst])) worst = i;
            if (ctas[worst] >= v[base + worst].a.n_tiles) break;
            ctas[worst]++;
        }
        FlowBatchArgs b;
        std::memset(static_cast<void *>(&b), 0, sizeof(b));
        size_t smem = 0;
        for (size_t i = 0; i < n; i++) {
            b.jobs[i] = v[base + i].a;
            b.variant[i] = v[base + i].variant;
            b.cta_begin[i + 1] = b.cta_begin[i] + ctas[i];
            smem = std::max(smem, v[base + i].j->shape.smem);
        }
        b.n_jobs = uint32_t(n);
        const cudaError_t e = flow_batch_launch(b, v[base].j->shape.threads, smem, st);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t flow_launch(const SigProgram &G, uint32_t n_obs, const DeviceSig *ds, const FlowShape &s,
                        const FlowCall &call, int sms, cudaStream_t st) {
    if (!ds || s.sched < 0 || size_t(s.sched) >= G.sched.size() || !ds->rows[s.sched]) return cudaErrorInvalidValue;
    const SigSchedule &S = G.sched[s.sched];
    FlowArgs a = flow_args(G, n_obs, ds, s, call);
    // tensor-store flush: by default for tiles of 8 or more chunks (rows of
    // 64 bytes or more; narrower boxes measured slower than plain stores);
    // TMCS_FLOW_TMA=1 for any even tile, 0 never; TMCS_FLOW_TMA_ROWS sets
    // the rows per box (default 64, rounded up to whole 128-byte stretches
    // of the ring)
    const uint32_t al = s.K >= 16 ? 1u : 16u / uint32_t(std::max(s.K, 1));
    const uint32_t trows = (uint32_t(std::max(env_int_flow("TMCS_FLOW_TMA_ROWS", 64), 1)) + al - 1) / al * al;
    const int tma = env_int_flow("TMCS_FLOW_TMA", -1);
    if ((tma > 0 || (tma < 0 && s.K >= 8)) && encode_det_map(&a.tmap, call.det, G.n_det, a.ld, s.K, trows))
        a.tma_rows = trows;
    // A CTA counts its batches and its steps in 32 bits: a call with more
    // tiles per CTA than that allows runs as several launches over column
    // slices (each a multiple of the tile size, in column order).
    const uint64_t per_tile_batches = batches_per_tile(S, s.K);
    const uint64_t per_tile_steps = a.n_steps;
    const uint64_t lim = (uint64_t(1) << 31) - 1;
    const uint64_t max_tiles_per_cta =
        std::max<uint64_t>(1, std::min(lim / std::max<uint64_t>(per_tile_batches, 1), lim / per_tile_steps) - 1);
    uint64_t slice_cols = max_tiles_per_cta * uint64_t(sms) * uint64_t(s.K);
    // testing knob: slices of this many tiles (so the sliced path runs at
    // sizes the tests can check)
    const int tslice = env_int_flow("TMCS_TEST_FLOW_SLICE_TILES", 0);
    if (tslice > 0) slice_cols = std::min<uint64_t>(slice_cols, uint64_t(tslice) * uint64_t(s.K));
    for (uint64_t c0 = 0; c0 < call.n_cols; c0 += slice_cols) {
        const uint64_t n = std::min(slice_cols, call.n_cols - c0);
        flow_columns(a, s, call, c0, n);
        cudaError_t e;
        switch (s.K) {
        case 16: e = flow_go_16(a, s, G.wide, sms, st); break;
        case 8: e = flow_go_8(a, s, G.wide, sms, st); break;
        case 4: e = flow_go_4(a, s, G.wide, sms, st); break;
        case 2: e = flow_go_2(a, s, G.wide, sms, st); break;
        default: e = flow_go_1(a, s, G.wide, sms, st); break;
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace tmcs
