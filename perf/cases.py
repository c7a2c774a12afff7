"""Sampling workloads and how to run one pass of each through the public API.

A case names a circuit of the distributed-QEC family (code, operation, rounds,
noise), the call made on it and the number of shots:

* ``sample``: ``Sampler.sample`` -- detector and observable words of a run;
* ``range``: the same with a first chunk, one slice of a long shot stream that
  a program consumes slice by slice;
* ``measurements``: raw measurement records;
* ``faults``: the signatures of a range of single faults, half of them
  (detector error model, extracted shard by shard);
* ``batch``: many small circuits in one ``tmcs_batch_sample`` call.

Compiled circuits are kept for the life of the process, as a sampling program
keeps them; seeds and output buffers are per call.
"""
import collections
import random

import torch

from paper_2504_05611_gb300 import circuits as C
from paper_2504_05611_gb300 import tmcs


def _case(name, call, code, op, rounds, p, p_ebit, shots, **more):
    return dict({"name": name, "call": call, "code": code, "op": op, "before": rounds[0], "after": rounds[1],
                 "p": p, "p_ebit": p_ebit, "shots": shots}, **more)


def listed():
    return [
        # the smallest call: a distance-3 non-local CNOT at its 1e4 shots
        # (threshold scans make thousands of these); launch and host latency
        _case("nl_sc3_1e4", "sample", "sc3", "nl", (3, 3), 1e-3, 1e-2, 10_000),
        # an ordinary point of a logical-error scan: distance 11, 1e5 shots,
        # a shot count that is no multiple of 64
        _case("nl_sc11_1e5", "sample", "sc11", "nl", (11, 11), 1e-3, 1e-2, 100_003),
        # a deep point of the same scan: the 1e7 shots a low error rate needs
        _case("nl_sc11_1e7", "sample", "sc11", "nl", (11, 11), 1e-3, 1e-2, 10_000_000),
        # the decoherence study: aged ebits carry PAULI_CHANNEL_1 noise
        _case("nl_sc11_deco_1e6", "sample", "sc11", "nl", (11, 11), 1e-3, 1e-3, 1_000_037, deco=1e-4),
        # BB[[144,12,12]] teleportation, 12 observables, weight-6 checks
        _case("tp_bb144_3e6", "sample", "bb144", "teleport", (12, 12), 1e-3, 1e-2, 3_000_000),
        # weight-4 Pauli string over five BB144 blocks, 60 observables
        _case("ps4_bb144_1e6", "sample", "bb144", "pauli4", (4, 1), 5e-4, 5e-4, 1_000_000),
        # the largest circuit (49,560 detectors) at the noise of the paper's
        # plots; a few GB of output per call
        _case("nl_sc29_2e6", "sample", "sc29", "nl", (29, 29), 1e-3, 1e-2, 2_000_000),
        # the same circuit at low noise, ragged: the output dominates
        _case("nl_sc29_low_2e6", "sample", "sc29", "nl", (29, 29), 1e-4, 1e-3, 1_999_981),
        # one 256 MiB slice of a stream of shots, as a program that copies
        # its results to the host slice by slice asks for
        _case("nl_sc29_slice", "range", "sc29", "nl", (29, 29), 1e-3, 1e-2, 677 * 64, first=1354),
        # 32 small circuits in one call (a parameter scan in one launch)
        _case("batch_small_32", "batch", "sc3-sc9", "mix", (0, 0), 1e-3, 1e-2, 0, jobs=32, mix=3),
        # raw measurement records for a program that forms its own detectors
        _case("meas_sc11_1e5", "measurements", "sc11", "nl", (11, 11), 1e-3, 1e-2, 100_000),
        # detector error model extraction, shard by shard: the signatures of
        # half of the circuit's single faults from some first one
        _case("faults_sc11", "faults", "sc11", "nl", (11, 11), 1e-3, 1e-2, 0),
    ]


_MAX_BYTES = 12_390_000_000  # output of the largest listed case


def _log(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng: random.Random):
    call = rng.choice(["sample", "sample", "sample", "sample", "range", "measurements", "faults", "batch"])
    if call == "batch":
        return {k: v for k, v in _case("", "batch", "sc3-sc9", "mix", (0, 0), 1e-3, 1e-2, 0, jobs=rng.randint(8, 32),
                                       mix=rng.randint(10, 10_000)).items() if k != "name"}
    small = call in ("measurements", "faults")
    code = rng.choice([f"sc{d}" for d in range(3, 12 if small else 30, 2)] + ["bb144"])
    d = 12 if code == "bb144" else int(code[2:])
    op = rng.choice(["nl", "teleport"])
    if code == "bb144" and rng.random() < 0.34:
        op = f"pauli{rng.randint(2, 4)}"
    p = _log(rng, 1e-4, 1e-3)
    ratio = rng.choice([1.0, 10.0])
    rounds = (rng.randint(2, 5), 1) if op.startswith("pauli") else (d, rng.choice([d, max(1, d - 1)]))
    # an upper bound of the output rows of any of these operations, so that a
    # drawn case stays below the largest listed one
    rows = 6 * (sum(rounds) + 2) * d * d + 64 if code != "bb144" else 20_000
    if call == "sample":
        top = max(20_000, min(10_000_000, int(8 * _MAX_BYTES / rows)))
        shots = int(_log(rng, 5_000, top)) + rng.randint(0, 63)
    elif call == "range":
        shots = 64 * max(8, min(2048, int(268_435_456 / (8 * rows)))) + rng.choice([0, 0, rng.randint(1, 63)])
    elif call == "measurements":
        shots = int(_log(rng, 5_000, 200_000))
    else:
        shots = 0
    c = _case("", call, code, op, rounds, p, ratio * p, shots)
    if call == "range":
        c["first"] = rng.randint(1, 100_000)
    if code != "bb144" and op == "nl" and rng.random() < 0.25:
        c["deco"] = _log(rng, 1e-5, 1e-3)
    del c["name"]
    return c


def _circuit(code, op, before, after, p, p_ebit, deco=0.0):
    noise = C.NoiseModel(p=p, p_ebit=p_ebit, decoherence=C.Decoherence(deco, schedule="lines") if deco else None)
    cc = C.code_by_name(code)
    if op == "nl":
        return C.nonlocal_cnot_circuit(cc, before, after, noise)
    if op == "teleport":
        return C.teleport_circuit(cc, before, after, noise)
    return C.pauli_string_circuit(cc, int(op[5:]), rounds_before=before, noise=noise)


# compiled circuits, the most recently used last
_SAMPLERS = collections.OrderedDict()
_KEPT = 160


def _sampler(use, spec):
    key = (use, spec)
    if key in _SAMPLERS:
        _SAMPLERS.move_to_end(key)
        return _SAMPLERS[key]
    s = _SAMPLERS[key] = tmcs.Sampler(_circuit(*spec))
    while len(_SAMPLERS) > _KEPT:
        _SAMPLERS.popitem(last=False)
    return s


def _spec(case):
    return (case["code"], case["op"], case["before"], case["after"], case["p"], case["p_ebit"], case.get("deco", 0.0))


def _batch_specs(case):
    """The circuits and shots of a batch: surface codes of distance 3 to 9,
    1e4 to 1e5 shots each."""
    rng = random.Random(case["mix"])
    out = []
    for j in range(case["jobs"]):
        d = rng.choice([3, 5, 7, 9])
        p = rng.choice([1e-4, 3e-4, 1e-3])
        out.append(((f"sc{d}", ("nl", "teleport")[j % 2], d, d, p, 10 * p, 0.0), int(round(_log(rng, 1e4, 1e5)))))
    return out


def _buffers(s, shots, rows=None):
    cols = (shots + 63) // 64
    if rows is not None:
        return torch.empty((rows, cols), dtype=torch.int64, device="cuda")
    return s.alloc(shots)


def prepare(case, seed):
    seed = (int(seed) * 0x9E3779B97F4A7C15 + 1) % 2 ** 63
    if case["call"] == "batch":
        jobs, keep = [], []
        for j, (spec, shots) in enumerate(_batch_specs(case)):
            s = _sampler("batch", spec)
            det, obs = _buffers(s, shots)
            jobs.append((s.handle, shots, (seed + j) % 2 ** 63, det, obs))
            keep.append(s)
        return {"call": "batch", "jobs": jobs, "keep": keep}
    s = _sampler((case["call"], case["shots"]), _spec(case))
    st = {"call": case["call"], "s": s, "seed": seed, "shots": case["shots"], "first": case.get("first", 0)}
    if case["call"] == "measurements":
        st["out"] = _buffers(s, case["shots"], s.info["n_meas"])
    elif case["call"] == "faults":
        total = tmcs.tmcs_fault_count(s.handle)
        st["shots"] = total // 2
        # shards start at a multiple of 64 faults
        st["first"] = 64 * random.Random(seed).randint(0, (total - st["shots"]) // 64)
        st["out"] = s.alloc(st["shots"])
    else:
        st["out"] = _buffers(s, case["shots"])
    return st


def run(st):
    if st["call"] == "batch":
        tmcs.tmcs_batch_sample(st["jobs"])
        return [t for job in st["jobs"] for t in job[3:5]]
    s, out = st["s"], st["out"]
    if st["call"] == "measurements":
        tmcs.tmcs_sample_measurements(s.handle, 0, st["shots"], st["seed"], out)
        return out
    if st["call"] == "faults":
        tmcs.tmcs_fault_signatures(s.handle, st["first"], st["shots"], out[0], out[1])
        return list(out)
    return list(s.sample(st["shots"], st["seed"], first_chunk=st["first"], out=out))


def work(case):
    """Output bytes of one pass: the words are written once; a circuit and a
    seed are all that is read. The path has no floating-point work."""
    if case["call"] == "batch":
        total = 0
        for spec, shots in _batch_specs(case):
            i = _sampler("batch", spec).info
            total += 8 * (i["n_det"] + i["n_obs"]) * ((shots + 63) // 64)
        return {"bytes": total, "flops": 0}
    s = _sampler((case["call"], case["shots"]), _spec(case))
    if case["call"] == "measurements":
        return {"bytes": 8 * s.info["n_meas"] * ((case["shots"] + 63) // 64), "flops": 0}
    shots = tmcs.tmcs_fault_count(s.handle) // 2 if case["call"] == "faults" else case["shots"]
    return {"bytes": 8 * (s.info["n_det"] + s.info["n_obs"]) * ((shots + 63) // 64), "flops": 0}


def exact(case, seed):
    """Outputs are bits, equal or wrong: there is no rounding to measure."""
    return None
