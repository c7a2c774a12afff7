"""Shapes of untimed calls and batches whose steps fill the event arena.

At p = 1e-2 (above the codes' thresholds) one step of the largest ring draws
several shared-memory arenas full of events, and every event beyond its
step's region waits until the step is applied. Calls and batches that nothing
has been timed for take a smaller ring or tile there.
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


def noisy(p):
    return C.nonlocal_cnot_circuit(C.code_by_name("sc11"), 11, 11, C.NoiseModel(p, 10 * p))


def best(call):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    for _ in range(13):
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return min(times[3:])


@pytest.mark.parametrize("p", [3e-3, 1e-2])
def test_batch_costs_about_one_call(p):
    """Eight jobs in one batch against the same shots in one call, whose
    shape is timed (with the largest ring for the batch: 2.7 and 3.1 times)."""
    n, shots = 8, 30_016
    s = tmcs.Sampler(noisy(p))
    jobs = [(s.handle, shots, j, *s.alloc(shots)) for j in range(n)]
    out = s.alloc(n * shots)
    batch = best(lambda: tmcs.tmcs_batch_sample(jobs))
    single = best(lambda: s.sample(n * shots, 1, out=out))
    tmcs.tmcs_check_device()
    assert batch < 1.6 * single, (batch, single)
    s.close()


@pytest.mark.parametrize("p", [3e-3, 1e-2])
def test_untimed_call_costs_about_its_share(p):
    """1,216 chunks on a fresh handle against a timed call of 3,752 chunks."""
    small, large = 1216 * 64, 3752 * 64
    s, t = tmcs.Sampler(noisy(p)), tmcs.Sampler(noisy(p))
    a, b = s.alloc(small), t.alloc(large)
    share = best(lambda: t.sample(large, 1, out=b)) * small / large
    untimed = best(lambda: s.sample(small, 1, out=a))
    tmcs.tmcs_check_device()
    assert untimed < 1.6 * share, (untimed, share)
    s.close()
    t.close()


@pytest.mark.parametrize("shots", [64 * 300 + 9, 64 * 1216])
def test_bits_equal_oracle(shots):
    """The shapes that the rule takes there, alone and in a batch."""
    circ = noisy(1e-2)
    s = tmcs.Sampler(circ)
    first = s.alloc(shots)
    s.sample(shots, 5, out=first)
    second = s.alloc(shots)
    tmcs.tmcs_batch_sample([(s.handle, shots, 5, *second)])
    torch.cuda.synchronize()
    tmcs.tmcs_check_device()
    cols = (shots + 63) // 64
    for col in (0, cols // 2, cols - 1):
        od, oo = oracle.sample(circ, min(64, shots - 64 * col), 5, first_chunk=col, threads=8)
        for det, obs in (first, second):
            assert np.array_equal(det[:, col].cpu().numpy().view(np.uint64), od[:, 0])
            assert np.array_equal(obs[: circ.n_obs, col].cpu().numpy().view(np.uint64), oo[:, 0])
    s.close()
