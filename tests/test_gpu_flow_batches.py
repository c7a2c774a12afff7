"""GPU parity of the decoupled kernel's batched walk with the CPU oracle.

A walker runs 32 streams (32 / K items x K chunks) through a first window of
Philox calls and puts the streams that go on aside in blocks of 32 (Methods
"Simulation": every draw of a stream is part of the sampled noise). The cases
sit at the edges: windows so short that nearly every stream goes on, blocks
that fill and overflow the step's space for them, steps whose items do not
fill a batch, chunk counts that do not fill a tile, and both slot layouts
(four rows per event, and eight for codes whose events flip many outputs).
The outputs are bits: they must equal the oracle's.
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


def check(monkeypatch, circ, shots, seed, first_chunk, **env):
    monkeypatch.setenv("TMCS_KERNEL", "7")
    for k, v in env.items():
        monkeypatch.setenv(k, str(v))
    s = tmcs.Sampler(circ)
    det, obs = s.sample(shots, seed, first_chunk=first_chunk)
    torch.cuda.synchronize()
    tmcs.tmcs_check_device()
    od, oo = oracle.sample(circ, shots, seed, first_chunk=first_chunk, threads=8)
    assert np.array_equal(det.cpu().numpy().view(np.uint64), od)
    assert np.array_equal(obs.cpu().numpy().view(np.uint64), oo)
    s.close()


@pytest.mark.parametrize("p", [2e-5, 1e-4, 1e-3, 4e-3])
@pytest.mark.parametrize("window,tile_k,cap", [(1, 8, 0), (1, 16, 0), (2, 4, 0), (4, 1, 0), (1, 8, 40)])
def test_streams_put_aside(monkeypatch, p, window, tile_k, cap):
    """Expected events per stream from 0.08 (one in 13 goes past a one-call
    window) to 16 (all do); cap: event regions of 40 entries, so that put-aside
    streams also meet full regions. p = 2e-5 needs the two-read gap count,
    which has no first window."""
    circ = C.nonlocal_cnot_circuit(C.code_by_name("sc7"), 5, 4, C.NoiseModel(p, 10 * p))
    env = dict(TMCS_FLOW_WINDOW=window, TMCS_TILE_K=tile_k, TMCS_SIG_SCHED=2)
    if cap:
        env["TMCS_TEST_FLOW_CAP"] = cap
    check(monkeypatch, circ, 64 * 53 + 17, 91, 7, **env)


@pytest.mark.parametrize("tile_k,threads,appliers", [(8, 1024, 30), (8, 96, 2), (16, 512, 4), (1, 64, 1)])
def test_eight_row_slots(monkeypatch, tile_k, threads, appliers):
    """BB[[18,4,4]] teleportation: events that flip up to eight outputs
    inline and longer lists, with many and few walker warps."""
    circ = C.teleport_circuit(C.code_by_name("bb18"), 2, 2, C.NoiseModel(0.004, 0.03))
    check(monkeypatch, circ, 64 * 41 + 1, 12, 3, TMCS_TILE_K=tile_k, TMCS_THREADS=threads, TMCS_FLOW_APPLIERS=appliers,
          TMCS_SIG_SCHED=2)


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 129])
@pytest.mark.parametrize("tile_k", [1, 8, 16])
def test_partial_batches(monkeypatch, n, tile_k):
    """One noise op of n units: steps of one to three items, fewer than a
    batch holds, with one column or a ragged last tile."""
    c = C.Circuit()
    q = list(range(n))
    c.append("R", q)
    c.append("X_ERROR", q, p=0.05)
    for r in c.append("M", q):
        c.append("DETECTOR", [int(r)])
    for shots in (1, 64 * 9 + 3):
        check(monkeypatch, c, shots, 5, 2, TMCS_TILE_K=tile_k)
