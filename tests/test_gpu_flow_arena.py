"""The decoupled kernel with an event arena smaller than its steps' events.

Steps are gated on the appliers and their regions clamped to the arena, for
every ring, with one and with several tiles per CTA; the bits are the
oracle's.
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


@pytest.mark.parametrize("sched,tile_k,appliers,arena,cap", [(0, 4, 8, 1024, 0), (0, 2, 4, 2048, 0), (2, 16, 8, 1024, 0),
                                                             (1, 8, 8, 1024, 3), (0, 1, 2, 1024, 0)])
def test_one_tile_per_cta(monkeypatch, sched, tile_k, appliers, arena, cap):
    circ = C.nonlocal_cnot_circuit(C.code_by_name("sc11"), 11, 11, C.NoiseModel(0.003, 0.02))
    env = {"TMCS_TEST_FLOW_CAP": cap} if cap else {}
    check(monkeypatch, circ, 64 * 19 + 45, 29, 3, TMCS_SIG_SCHED=sched, TMCS_TILE_K=tile_k, TMCS_FLOW_APPLIERS=appliers,
          TMCS_FLOW_ARENA=arena, **env)


@pytest.mark.parametrize("tile_k,arena", [(8, 1024), (8, 4096), (2, 1024)])
def test_many_tiles_per_cta(monkeypatch, tile_k, arena):
    circ = C.nonlocal_cnot_circuit(C.code_by_name("sc5"), 6, 6, C.NoiseModel(0.01, 0.05))
    check(monkeypatch, circ, 64 * 2002 - 5, 41, 11, TMCS_TILE_K=tile_k, TMCS_FLOW_ARENA=arena)
