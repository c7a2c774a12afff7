"""Batched sampling through the decoupled kernel: many circuits in one launch.

Every job has CTAs of its own in the shared launch, one launch per kernel
variant (two slot layouts; tables in shared memory without PAULI_CHANNEL_1, or
the general kernel) and per 64 jobs. Each job's bits must equal the oracle's
(Methods "Simulation"; a batch changes only where a circuit runs): mixed
variants, one column, ragged columns, more jobs than a launch holds, regions
too small for their events.
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


def circuits():
    sc3, sc5, bb = C.code_by_name("sc3"), C.code_by_name("sc5"), C.code_by_name("bb18")
    return [
        C.nonlocal_cnot_circuit(sc3, 3, 3, C.NoiseModel(1e-3, 1e-2)),
        C.teleport_circuit(sc5, 2, 2, C.NoiseModel(0.01, 0.05)),
        C.teleport_circuit(bb, 1, 1, C.NoiseModel(0.004, 0.03)),  # eight rows per slot
        C.nonlocal_cnot_circuit(sc5, 2, 2, C.NoiseModel(0.003, 0.02, decoherence=C.Decoherence(0.05))),
        C.nonlocal_cnot_circuit(sc3, 2, 2, C.NoiseModel(1e-5, 1e-4)),  # two-read gap counts
    ]


@pytest.mark.parametrize("shots", [(1, 64, 65, 64 * 9 + 3, 64 * 700 + 1), (64 * 4, 64 * 5, 64 * 611, 63, 129)])
@pytest.mark.parametrize("repeat,cap", [(1, 0), (15, 0), (1, 3)])
def test_jobs_equal_oracle(monkeypatch, shots, repeat, cap):
    if cap:
        monkeypatch.setenv("TMCS_TEST_FLOW_CAP", str(cap))
    circs = circuits()
    samplers = [tmcs.Sampler(c) for c in circs]
    jobs, want = [], []
    for r in range(repeat):
        for i, (c, s) in enumerate(zip(circs, samplers)):
            n = shots[i] if r == 0 else min(shots[i], 200)
            det, obs = s.alloc(n)
            det.fill_(-1)
            obs.fill_(-1)
            jobs.append((s.handle, n, 100 * r + i, det, obs))
            want.append((c, n, 100 * r + i))
    tmcs.tmcs_batch_sample(jobs)
    torch.cuda.synchronize()
    tmcs.tmcs_check_device()
    for (c, n, seed), job in zip(want, jobs):
        od, oo = oracle.sample(c, n, seed, threads=8)
        assert np.array_equal(job[3].cpu().numpy().view(np.uint64), od)
        assert np.array_equal(job[4][: c.n_obs].cpu().numpy().view(np.uint64), oo)
    for s in samplers:
        s.close()
