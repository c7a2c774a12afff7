"""The reported first window of the decoupled kernel is the one that runs.

The general kernel (here for PAULI_CHANNEL_1 noise, Methods "Decoherence") has
windows of one and three calls; a request for two or four runs three.
"""
import pytest

from paper_2504_05611_gb300 import circuits as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_05611_gb300 import tmcs  # noqa: E402


@pytest.mark.parametrize("deco,asked,runs", [(0.01, 1, 1), (0.01, 2, 3), (0.01, 3, 3), (0.01, 4, 3),
                                             (0.0, 1, 1), (0.0, 2, 2), (0.0, 4, 4)])
def test_reported_window(monkeypatch, deco, asked, runs):
    monkeypatch.setenv("TMCS_FLOW_WINDOW", str(asked))
    noise = C.NoiseModel(1e-3, 1e-2, decoherence=C.Decoherence(deco) if deco else None)
    s = tmcs.Sampler(C.nonlocal_cnot_circuit(C.code_by_name("sc3"), 2, 2, noise))
    s.sample(64 * 152 * 16, 1)  # large enough to be timed
    torch.cuda.synchronize()
    shape = tmcs.tmcs_launch_shape(s.handle)
    assert shape["mode"] == 7 and shape["window"] == runs
    s.close()
