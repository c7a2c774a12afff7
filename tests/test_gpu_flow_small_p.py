"""Noise ops of very small p next to ordinary ones in the decoupled kernel.

A gap table of p below about 2.1e-5 needs the two-read gap count. Which count
a walker uses is a choice per batch of 32 streams: a few such ops (aged ebits
after a short wait, Methods "Decoherence") change neither the bits of a
program nor the time of its other streams.
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


def mixed_circuit(n):
    """Readout of n qubits after noise of p = 1e-5 and of ordinary p, so that
    a step holds segments of both kinds, alone and in one batch."""
    c = C.Circuit()
    q = list(range(n))
    c.append("R", q)
    c.append("X_ERROR", q, p=1e-5)
    c.append("DEPOLARIZE1", q, p=0.02)
    c.append("X_ERROR", q[: n // 2 + 1], p=1.5e-5)
    c.append("X_ERROR", q, p=3e-3)
    for r in c.append("M", q):
        c.append("DETECTOR", [int(r)])
    return c


def decoherence_circuit(code, rounds, deco, p=1e-3):
    nz = C.NoiseModel(p=p, p_ebit=p, decoherence=C.Decoherence(deco, schedule="lines"))
    return C.nonlocal_cnot_circuit(C.code_by_name(code), rounds, rounds, nz)


CASES = {"n1": lambda: mixed_circuit(1), "n65": lambda: mixed_circuit(65), "n700": lambda: mixed_circuit(700),
         "sc5": lambda: decoherence_circuit("sc5", 3, 1e-5), "sc7": lambda: decoherence_circuit("sc7", 4, 2e-5, 4e-3),
         "bb18": lambda: decoherence_circuit("bb18", 2, 1e-5, 4e-3)}


@pytest.mark.parametrize("case", list(CASES))
@pytest.mark.parametrize("window,tile_k,cap", [(1, 1, 0), (1, 8, 0), (3, 8, 0), (3, 16, 0), (1, 4, 7)])
def test_bits_equal_oracle(monkeypatch, case, window, tile_k, cap):
    monkeypatch.setenv("TMCS_KERNEL", "7")
    monkeypatch.setenv("TMCS_FLOW_WINDOW", str(window))
    monkeypatch.setenv("TMCS_TILE_K", str(tile_k))
    monkeypatch.setenv("TMCS_SIG_SCHED", "2")
    if cap:
        monkeypatch.setenv("TMCS_TEST_FLOW_CAP", str(cap))
    circ = CASES[case]()
    shots, seed, first = 64 * 53 + 17, 19, 5
    s = tmcs.Sampler(circ)
    det, obs = s.sample(shots, seed, first_chunk=first)
    torch.cuda.synchronize()
    tmcs.tmcs_check_device()
    od, oo = oracle.sample(circ, shots, seed, first_chunk=first, threads=8)
    assert np.array_equal(det.cpu().numpy().view(np.uint64), od)
    assert np.array_equal(obs.cpu().numpy().view(np.uint64)[: circ.n_obs], oo)
    s.close()


def best_time(circ, shots):
    s = tmcs.Sampler(circ)
    out = s.alloc(shots)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    for seed in range(23):
        a.record()
        s.sample(shots, seed, out=out)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    s.close()
    return min(times[3:])


def test_small_p_does_not_slow_the_other_ops():
    """d=11 with two decoherence strengths, one just below and one just above
    the limit: the same ops with nearly the same work, so the same time (when
    one such op took the first window from the whole program: 1.47 times)."""
    below = best_time(decoherence_circuit("sc11", 11, 2e-5), 1_000_000)
    above = best_time(decoherence_circuit("sc11", 11, 3e-5), 1_000_000)
    assert below < 1.2 * above, (below, above)
