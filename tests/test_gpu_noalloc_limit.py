"""The size limit of the allocation-free entry point.

The limit is 8 MiB for the compiled program without the records that apply
its noise ops' events: a program of many small noise ops, each applied by a
layer of its own, has about as many bytes of records again.
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


def many_small_ops(n):
    """n single-qubit flips with a CX after each (so that no two share a
    layer): 118 bytes a flip, and 28 of records."""
    c = C.Circuit()
    c.append("R", [0, 1, 2, 3])
    for i in range(n):
        c.append("X_ERROR", [0], p=2e-4)
        c.append("CX", [i % 4, (i + 1) % 4])
    for r in c.append("M", [0, 1, 2, 3]):
        c.append("DETECTOR", [int(r)])
    return c


def test_program_of_many_records_is_taken():
    circ = many_small_ops(70_000)  # 8.28 MB, and 1.96 MB of records
    h = tmcs.tmcs_circuit_build(circ)
    shots, seed = 64 * 3 + 5, 17
    det = torch.full((4, 4), -1, dtype=torch.int64, device="cuda")
    obs = torch.empty((1, 4), dtype=torch.int64, device="cuda")
    tmcs.tmcs_sample_noalloc(h, 0, shots, seed, det, obs)
    torch.cuda.synchronize()
    tmcs.tmcs_check_device()
    want, _ = oracle.sample(circ, shots, seed, threads=8)
    assert np.array_equal(det.cpu().numpy().view(np.uint64), want)
    tmcs.tmcs_circuit_free(h)


def test_program_above_the_limit_is_refused():
    h = tmcs.tmcs_circuit_build(many_small_ops(72_000))  # 8.51 MB without the records
    det = torch.zeros((4, 1), dtype=torch.int64, device="cuda")
    with pytest.raises(tmcs.TmcsError) as e:
        tmcs.tmcs_sample_noalloc(h, 0, 64, 1, det, det)
    assert e.value.code == 1 and "at most" in str(e.value)
    tmcs.tmcs_circuit_free(h)
