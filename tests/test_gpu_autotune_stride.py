"""The autotuner times the shapes at the row stride of the call it tunes for.

The low-noise d=29 circuit at 1e7 shots is bound by its writes, 32 or 64
bytes per row and tile at a stride of 1.25 MB: tiles of eight chunks take
26.6 ms and tiles of four 32.9, which a compact output of the timed columns
did not show.
"""
import pytest

from paper_2504_05611_gb300 import circuits as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_05611_gb300 import tmcs  # noqa: E402


def best(s, shots, out):
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    times = []
    for seed in range(6):
        a.record()
        s.sample(shots, seed, out=out)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return min(times[2:])


def test_wide_stride(monkeypatch):
    shots = 10_000_000
    s = tmcs.Sampler(C.nonlocal_cnot_circuit(C.code_by_name("sc29"), 29, 29, C.NoiseModel(1e-4, 1e-3)))
    out = s.alloc(shots)
    tuned = best(s, shots, out)
    for k, v in {"TMCS_KERNEL": "7", "TMCS_TILE_K": "8", "TMCS_SIG_SCHED": "1", "TMCS_FLOW_APPLIERS": "12"}.items():
        monkeypatch.setenv(k, v)
    forced = best(s, shots, out)
    tmcs.tmcs_check_device()
    assert tuned < 1.12 * forced, (tuned, forced)
    s.close()
    del out
    torch.cuda.empty_cache()
