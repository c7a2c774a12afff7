// Every interleaving of walkers and appliers over the step completion code of
// the decoupled kernel (csrc/tmcs_flow_step.h), on the CPU.
//
// One slot, two steps that use it one after the other, two walkers, one
// applier. Each access to shared state is one atomic action (the kernel's
// are at least as ordered: acquire, release, warp and CTA barriers). A thread
// is run again from its start with the results of its earlier actions, so a
// state is the shared memory and the threads' results; all states are
// visited. Checked: a block of put-aside streams is finished only while its
// step is the one in the slot, and once; a step is applied only when all its
// streams are finished; every state can still reach the end.
#include <cstdint>
#include <cstdio>
#include <unordered_map>
#include <string>
#include <vector>

#include "tmcs_flow_step.h"

namespace {

constexpr uint32_t kLcap = 64;  // room for put-aside streams: two blocks
using Steps = std::vector<std::vector<uint32_t>>;  // streams put aside by every batch of every step

struct Shared {
    uint32_t next = 0, applied = 0, done = 0, left = 0;
    uint32_t blk[2] = {};
    uint32_t finished[2] = {};  // per step: bit b = block b finished
};

struct Yield {};
struct Bad {
    const char *what;
};

struct Thread {
    std::vector<uint32_t> log;
    bool ended = false;
};

struct Run {
    Shared &m;
    std::vector<uint32_t> &log;
    const Steps &steps;
    size_t at = 0;
    bool acted = false;
    template <class F>
    uint32_t act(F &&f) {
        if (at < log.size()) return log[at++];
        if (acted) throw Yield{};
        acted = true;
        log.push_back(f());
        return log[at++];
    }
    // polls until cond() holds; a poll that fails leaves no trace
    template <class C>
    void poll(C &&cond) {
        const size_t start = at;
        if (!cond()) {
            log.resize(start);
            throw Yield{};
        }
    }
};

struct Slot {
    Run &r;
    uint32_t add_batch() {
        return r.act([&]() { return (r.m.done += 1u) - 1u; });
    }
    void add_unit() {
        r.act([&]() { return r.m.done += 0x10000u; });
    }
    uint32_t done() {
        return r.act([&]() { return r.m.done; });
    }
    uint32_t left() {
        return r.act([&]() { return r.m.left; });
    }
};

// Streams that a step leaves in its region.
uint32_t kept(const std::vector<uint32_t> &step) {
    uint32_t n = 0;
    for (uint32_t a : step) n += a;
    return n < kLcap ? n : kLcap;
}

void finish(Run &r, uint32_t Q, uint32_t blk, uint32_t n) {
    r.act([&]() -> uint32_t {
        if (r.m.applied != Q) throw Bad{"block finished after its step was applied"};
        const uint32_t k = kept(r.steps[Q]);
        if (blk > 1 || 32 * blk >= k || n != (k - 32 * blk < 32 ? k - 32 * blk : 32u)) throw Bad{"wrong block"};
        if (r.m.finished[Q] >> blk & 1u) throw Bad{"block finished twice"};
        return r.m.finished[Q] |= 1u << blk;
    });
}

void walker(Run &r) {
    uint32_t total = 0;
    for (const auto &s : r.steps) total += uint32_t(s.size());
    for (;;) {
        const uint32_t g = r.act([&]() { return r.m.next++; });
        if (g >= total) return;
        uint32_t Q = 0, b = g;
        while (b >= r.steps[Q].size()) b -= uint32_t(r.steps[Q++].size());
        const uint32_t nb = uint32_t(r.steps[Q].size());
        r.poll([&]() { return r.act([&]() { return r.m.applied; }) == Q; });
        bool full[2] = {};
        if (const uint32_t n = r.steps[Q][b]) {
            const uint32_t base = r.act([&]() { return (r.m.left += n) - n; });
            const uint32_t hi = base + n < kLcap ? base + n : kLcap;
            for (uint32_t k = 0; k < 2; k++) {
                const uint32_t f = base > 32 * k ? base : 32 * k, e = hi < 32 * k + 32 ? hi : 32 * k + 32;
                if (f < e) full[k] = r.act([&]() { return r.m.blk[k] += e - f; }) == 32;
            }
        }
        Slot s{r};
        tmcs::flow_batch_walked(
            s, nb, kLcap,
            [&]() {
                for (uint32_t k = 0; k < 2; k++)
                    if (full[k]) {
                        finish(r, Q, k, 32);
                        s.add_unit();
                    }
            },
            [&](uint32_t blk, uint32_t n) { finish(r, Q, blk, n); });
    }
}

void applier(Run &r) {
    for (uint32_t Q = 0; Q < r.steps.size(); Q++) {
        Slot s{r};
        r.poll([&]() { return tmcs::flow_step_complete(s, uint32_t(r.steps[Q].size()), kLcap); });
        r.act([&]() -> uint32_t {
            const uint32_t k = kept(r.steps[Q]);
            if (r.m.finished[Q] != (1u << ((k + 31) / 32)) - 1u) throw Bad{"step applied before its streams ended"};
            return 0;
        });
        r.act([&]() { return r.m.done = 0; });
        r.act([&]() { return r.m.left = 0; });
        r.act([&]() { return r.m.blk[0] = r.m.blk[1] = 0; });
        r.act([&]() { return r.m.applied = Q + 1; });
    }
}

struct State {
    Shared m;
    Thread t[3];  // two walkers, the applier
    std::string key() const {
        std::string k(reinterpret_cast<const char *>(&m), sizeof(m));
        for (const Thread &x : t) {
            k += char(x.ended);
            k += char(x.log.size());
            for (uint32_t v : x.log) k.append(reinterpret_cast<const char *>(&v), 4);
        }
        return k;
    }
};

// Number of states, or 0 with the reason printed.
size_t explore(const Steps &steps) {
    std::unordered_map<std::string, size_t> id;
    std::vector<State> states;
    std::vector<std::vector<size_t>> from;
    std::vector<size_t> ends;
    auto add = [&](const State &s) {
        const auto ins = id.emplace(s.key(), states.size());
        if (ins.second) {
            states.push_back(s);
            from.emplace_back();
        }
        return ins.first->second;
    };
    add(State{});
    for (size_t i = 0; i < states.size(); i++) {
        bool all = true;
        for (int k = 0; k < 3; k++) {
            if (states[i].t[k].ended) continue;
            all = false;
            State n = states[i];
            try {
                Run r{n.m, n.t[k].log, steps};
                if (k < 2) walker(r);
                else applier(r);
                n.t[k].ended = true;
            } catch (const Yield &) {
            } catch (const Bad &b) {
                std::printf("%s\n", b.what);
                return 0;
            }
            from[add(n)].push_back(i);
        }
        if (all) ends.push_back(i);
    }
    std::vector<char> reach(states.size(), 0);
    while (!ends.empty()) {
        const size_t i = ends.back();
        ends.pop_back();
        if (reach[i]) continue;
        reach[i] = 1;
        for (size_t p : from[i]) ends.push_back(p);
    }
    for (char c : reach)
        if (!c) {
            std::printf("a state that cannot end\n");
            return 0;
        }
    return states.size();
}

}  // namespace

int main() {
    const Steps kinds = {{0}, {5}, {32}, {0, 0}, {5, 0}, {20, 12}, {32, 3}, {32, 32}};
    size_t n = 0;
    for (const auto &a : kinds)
        for (const auto &b : kinds) {
            const size_t k = explore({a, b});
            if (!k) {
                std::printf("first step:");
                for (uint32_t x : a) std::printf(" %u", x);
                std::printf(", second step:");
                for (uint32_t x : b) std::printf(" %u", x);
                std::printf("\n");
                return 1;
            }
            n += k;
        }
    // more streams than the region holds: the rest is finished in place
    if (!explore({{30, 30, 30}, {30, 2}})) return 1;
    std::printf("%zu states\n", n);
    return 0;
}
