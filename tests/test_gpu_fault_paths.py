"""Fault signatures by every route (Methods "Decoding": a detector error model
column per fault).

By default they are scattered from the event table; the frame program injects
them where that table is not on the device and cannot be brought there, as
while a stream is being captured, or when its kernel is asked for.
"""
import numpy as np
import pytest

from paper_2504_05611_gb300 import circuits as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_05611_gb300 import tmcs  # noqa: E402


def circuit():
    return C.nonlocal_cnot_circuit(C.code_by_name("sc5"), 2, 2, C.NoiseModel(0.003, 0.02,
                                                                             decoherence=C.Decoherence(0.01)))


def signatures(s, first, n, out=None):
    det, obs = out if out is not None else s.alloc(n)
    tmcs.tmcs_fault_signatures(s.handle, first, n, det, obs)
    return det, obs


@pytest.mark.parametrize("env", [{"TMCS_KERNEL": "3"}, {"TMCS_KERNEL": "3", "TMCS_TILE_K": "2", "TMCS_THREADS": "64"},
                                 {"TMCS_KERNEL": "4"}])
@pytest.mark.parametrize("first,n", [(0, 1), (64, 1001), (0, None)])
def test_injection_equals_scatter(monkeypatch, env, first, n):
    s = tmcs.Sampler(circuit())
    n = n or tmcs.tmcs_fault_count(s.handle)
    want = [t.clone() for t in signatures(s, first, n)]
    with monkeypatch.context() as m:
        for k, v in env.items():
            m.setenv(k, v)
        got = signatures(s, first, n)
    torch.cuda.synchronize()
    tmcs.tmcs_check_device()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    assert bool(want[0].any())
    s.close()


@pytest.mark.parametrize("table", [False, True])
def test_captured_signatures(monkeypatch, table):
    """Captured on a handle whose frame program is on the device, without and
    with its event table."""
    s = tmcs.Sampler(circuit())
    other = tmcs.Sampler(circuit())
    n = tmcs.tmcs_fault_count(s.handle)
    want = signatures(other, 0, n)
    with monkeypatch.context() as m:
        m.setenv("TMCS_KERNEL", "3")
        s.sample(64, 1)
    if table:
        s.sample(64, 1)
    out = s.alloc(n)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        signatures(s, 0, n, out)
    for _ in range(2):
        for t in out:
            t.fill_(-1)
        g.replay()
        torch.cuda.synchronize()
        tmcs.tmcs_check_device()
        for a, b in zip(out, want):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
    del g
    s.close()
    other.close()
