"""Batches off the decoupled kernel.

The barrier signature kernel takes a batch that the decoupled kernel does not
fit (here by asking for it), in two size classes and in launches of at most
96 jobs; the frame kernel takes one with a circuit that has no signature
program. The bits are the oracle's either way.
"""
import numpy as np
import pytest

import oracle
from paper_2504_05611_gb300 import circuits as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_05611_gb300 import tmcs  # noqa: E402


def prepare(circs, shots):
    samplers = [tmcs.Sampler(c) for c in circs]
    jobs = []
    for i, (s, n) in enumerate(zip(samplers, shots)):
        det, obs = s.alloc(n)
        det.fill_(-1)
        obs.fill_(-1)
        jobs.append((s.handle, n, 300 + i, det, obs))
    return samplers, jobs


def check(circs, jobs):
    torch.cuda.synchronize()
    tmcs.tmcs_check_device()
    for c, (_, n, seed, det, obs) in zip(circs, jobs):
        od, oo = oracle.sample(c, n, seed, threads=8)
        assert np.array_equal(det.cpu().numpy().view(np.uint64), od)
        assert np.array_equal(obs[: c.n_obs].cpu().numpy().view(np.uint64), oo)


def mixed():
    """Jobs of both size classes: d=29 in the four-chunk one."""
    circs = [C.nonlocal_cnot_circuit(C.code_by_name("sc3"), 2, 2, C.NoiseModel(0.01, 0.05)),
             C.WORKLOADS["nl_sc29"].circuit(),
             C.teleport_circuit(C.code_by_name("bb18"), 1, 1, C.NoiseModel(0.004, 0.03)),
             C.nonlocal_cnot_circuit(C.code_by_name("sc5"), 2, 2,
                                     C.NoiseModel(0.003, 0.02, decoherence=C.Decoherence(0.05)))]
    return circs, [64 * 40 + 9, 64 * 2 + 5, 64 * 21, 64 * 11 + 63]


def many():
    code = C.code_by_name("sc3")
    circs = [C.nonlocal_cnot_circuit(code, 1 + i % 3, 1, C.NoiseModel(0.01, 0.05)) for i in range(110)]
    return circs, [1 + 37 * i for i in range(110)]


@pytest.mark.parametrize("kernel", ["5", "6"])
@pytest.mark.parametrize("case", [mixed, many])
def test_barrier_kernel(monkeypatch, kernel, case):
    monkeypatch.setenv("TMCS_KERNEL", kernel)
    circs, shots = case()
    samplers, jobs = prepare(circs, shots)
    tmcs.tmcs_batch_sample(jobs)
    check(circs, jobs)
    for s in samplers:
        s.close()


def test_barrier_kernel_in_a_graph(monkeypatch):
    monkeypatch.setenv("TMCS_KERNEL", "5")
    circs, shots = mixed()
    samplers, jobs = prepare(circs, shots)
    tmcs.tmcs_batch_sample(jobs)  # uploads the programs, makes the work queue
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        tmcs.tmcs_batch_sample(jobs)
    for _ in range(2):
        for job in jobs:
            job[3].fill_(-1)
            job[4].fill_(-1)
        g.replay()
        check(circs, jobs)
    del g
    for s in samplers:
        s.close()


def test_a_job_without_signature_program():
    """20,000 noise ops, more than the signature program's item records hold."""
    c = C.Circuit()
    c.append("R", [0, 1, 2, 3])
    for i in range(20_000):
        c.append("X_ERROR", [0], p=2e-4)
        c.append("CX", [i % 4, (i + 1) % 4])
    for r in c.append("M", [0, 1, 2, 3]):
        c.append("DETECTOR", [int(r)])
    circs, shots = mixed()
    circs, shots = [circs[0], c, circs[2]], [shots[0], 64 * 3 + 1, shots[2]]
    samplers, jobs = prepare(circs, shots)
    assert [tmcs.tmcs_circuit_stats(s.handle)["sig_ok"] for s in samplers] == [1, 0, 1]
    tmcs.tmcs_batch_sample(jobs)
    check(circs, jobs)
    for s in samplers:
        s.close()
