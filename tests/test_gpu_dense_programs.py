"""Programs of hundreds of events per noise stream (p of several percent).

Their steps do not fit the decoupled kernel's event arena, and the barrier
kernel is the faster one for them: untimed calls choose it by a rule, timed
calls by measuring both, and batches with such a job run it.
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


def dense(code="sc11", rounds=11, p=0.1):
    return C.nonlocal_cnot_circuit(C.code_by_name(code), rounds, rounds, C.NoiseModel(p, p))


def best(call):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    for _ in range(8):
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return min(times[3:])


@pytest.mark.parametrize("chunks", [1250, 4688])
def test_call_takes_the_faster_kernel(monkeypatch, chunks):
    """1,250 chunks by rule (decoupled kernel 3.8 ms, barrier 2.1), 4,688 by
    timing."""
    s = tmcs.Sampler(dense())
    out = s.alloc(64 * chunks)
    default = best(lambda: s.sample(64 * chunks, 1, out=out))
    monkeypatch.setenv("TMCS_KERNEL", "5")
    barrier = best(lambda: s.sample(64 * chunks, 1, out=out))
    tmcs.tmcs_check_device()
    assert default < 1.2 * barrier, (default, barrier)
    s.close()


def test_batch_takes_the_faster_kernel(monkeypatch):
    s = tmcs.Sampler(dense())
    jobs = [(s.handle, 20_000, j, *s.alloc(20_000)) for j in range(8)]
    default = best(lambda: tmcs.tmcs_batch_sample(jobs))
    monkeypatch.setenv("TMCS_KERNEL", "5")
    barrier = best(lambda: tmcs.tmcs_batch_sample(jobs))
    tmcs.tmcs_check_device()
    assert default < 1.2 * barrier, (default, barrier)
    s.close()


@pytest.mark.parametrize("code,rounds,p", [("sc11", 11, 0.1), ("sc7", 7, 0.2), ("sc5", 3, 0.4), ("bb18", 2, 0.2)])
@pytest.mark.parametrize("chunks", [3, 700])
def test_bits_equal_oracle(code, rounds, p, chunks):
    circ = dense(code, rounds, p)
    shots = 64 * chunks - 5
    s = tmcs.Sampler(circ)
    det, obs = s.sample(shots, 23)
    bdet, bobs = s.alloc(shots)
    tmcs.tmcs_batch_sample([(s.handle, shots, 23, bdet, bobs)])
    torch.cuda.synchronize()
    tmcs.tmcs_check_device()
    assert torch.equal(det, bdet) and torch.equal(obs, bobs)
    for col in (0, chunks // 2, chunks - 1):
        od, oo = oracle.sample(circ, min(64, shots - 64 * col), 23, first_chunk=col, threads=8)
        assert np.array_equal(det[:, col].cpu().numpy().view(np.uint64), od[:, 0])
        assert np.array_equal(obs[: circ.n_obs, col].cpu().numpy().view(np.uint64), oo[:, 0])
    s.close()
