"""The validator of the decoupled kernel's event classes and row tables (CPU).

Pauli indices of a segment that flip the same outputs in every unit share a
class, whose output rows each schedule stores once per unit. The program is
refused when an index is in a class with another output list, or when a row
differs from the list's.
"""
import pytest

from paper_2504_05611_gb300 import circuits as C
from paper_2504_05611_gb300 import tmcs


def circuit(code, deco=0.0):
    noise = C.NoiseModel(1e-3, 1e-2, decoherence=C.Decoherence(deco) if deco else None)
    return C.nonlocal_cnot_circuit(C.code_by_name(code), 3, 3, noise)


@pytest.mark.parametrize("code,deco", [("sc3", 0.0), ("sc7", 0.01), ("bb18", 0.0)])
@pytest.mark.parametrize("mistake,reason", [(None, None), ("class", "event class"), ("row", "event row")])
def test_planted_mistakes(monkeypatch, code, deco, mistake, reason):
    if mistake:
        monkeypatch.setenv("TMCS_TEST_CORRUPT_SIG", mistake)
    h = tmcs.tmcs_circuit_build(circuit(code, deco))
    try:
        assert tmcs.tmcs_circuit_stats(h)["sig_ok"] == (0 if mistake else 1)
        if mistake:
            with pytest.raises(tmcs.TmcsError) as err:
                tmcs.tmcs_fault_outputs(h, 0)
            assert "internal" in str(err.value) and reason in str(err.value)
    finally:
        tmcs.tmcs_circuit_free(h)
