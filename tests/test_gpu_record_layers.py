"""Layer grouping of the raw-measurement program and the single-fault scatter.

The measurement program emits an op's record outputs and gauge Paulis after
all its targets (Methods "Simulation": one noisy execution, one record per
measurement), except for circuits so wide that the grouped program's frame
words would not fit; both must give the oracle's records, also when an op
names a qubit twice. tmcs_fault_signatures writes a fault range by scattering
every fault's output list into a zeroed output; ranges are compared with the
frame program that injects one fault per lane. All outputs are bits: equal or
wrong.
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


def records(circ, shots, seed, first_chunk):
    h = tmcs.tmcs_circuit_build(circ, tmcs.TMCS_FLAG_NO_AUDIT)
    meas = torch.full((circ.n_meas, (shots + 63) // 64), -1, dtype=torch.int64, device="cuda")
    tmcs.tmcs_sample_measurements(h, first_chunk, shots, seed, meas)
    torch.cuda.synchronize()
    tmcs.tmcs_check_device()
    tmcs.tmcs_circuit_free(h)
    return meas.cpu().numpy().view(np.uint64)


@pytest.mark.parametrize("meas", ["M", "MX"])
@pytest.mark.parametrize("reset", ["R", "RX"])
def test_repeated_targets(meas, reset):
    c = C.Circuit()
    c.append(reset, [0, 1, 0, 2])
    c.append("DEPOLARIZE2", [0, 1], p=0.1)
    c.append("H", [1])
    c.append(meas, [0, 1, 0, 2, 1])
    c.append("CX", [0, 1, 1, 2])
    c.append("X_ERROR", [0, 1, 2], p=0.2)
    c.append(meas, [2, 2, 0])
    got = records(c, 64 * 3 + 5, 17, 4)
    assert np.array_equal(got, oracle.sample_measurements(c, 64 * 3 + 5, 17, first_chunk=4))


@pytest.mark.parametrize("n", [300, 20_400])
def test_wide_measurement_op(n):
    """n qubits measured by one op; 20,400 frame words exceed what the
    grouped layers may use, so the program is compiled target by target."""
    c = C.Circuit()
    q = list(range(n))
    c.append("R", q)
    c.append("X_ERROR", q, p=0.01)
    c.append("M", q)
    got = records(c, 64 + 9, 3, 1)
    ref = np.zeros(n, dtype=np.uint8)
    assert np.array_equal(got, oracle.sample_measurements(c, 64 + 9, 3, first_chunk=1, reference=ref))


@pytest.mark.parametrize("code,op", [("sc5", "nl"), ("bb18", "teleport")])
@pytest.mark.parametrize("lo,count", [(0, 1), (64, 63), (128, 64), (192, 65), (640, 2001), (0, None)])
def test_fault_ranges(monkeypatch, code, op, lo, count):
    fn = C.nonlocal_cnot_circuit if op == "nl" else C.teleport_circuit
    circ = fn(C.code_by_name(code), 2, 2, C.NoiseModel(0.003, 0.02))
    s = tmcs.Sampler(circ)
    n = tmcs.tmcs_fault_count(s.handle) - lo if count is None else count

    def run():
        det, obs = s.alloc(n)
        det.fill_(-1)
        obs.fill_(-1)
        tmcs.tmcs_fault_signatures(s.handle, lo, n, det, obs)
        torch.cuda.synchronize()
        return det.cpu().numpy(), obs[: circ.n_obs].cpu().numpy()

    got = run()
    monkeypatch.setenv("TMCS_KERNEL", "3")  # the frame program with injected faults
    want = run()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    assert got[0].any()
    s.close()
