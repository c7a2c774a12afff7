"""Jobs of different kinds share one batched launch of the decoupled kernel.

A surface code, a BB code (eight rows per event slot) and a circuit with ebit
decoherence (PAULI_CHANNEL_1 noise, Methods "Decoherence") each run another
variant of the kernel. With few columns a job's time is its chain of steps,
so jobs that run side by side take as long as the longest of them and not as
long as all of them together.
"""
import pytest

from paper_2504_05611_gb300 import circuits as C

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_05611_gb300 import tmcs  # noqa: E402


def test_kinds_run_side_by_side():
    circs = [C.nonlocal_cnot_circuit(C.code_by_name("sc15"), 15, 15, C.NoiseModel(1e-3, 1e-2)),
             C.teleport_circuit(C.code_by_name("bb144"), 12, 12, C.NoiseModel(1e-3, 1e-2)),
             C.nonlocal_cnot_circuit(C.code_by_name("sc15"), 15, 15,
                                     C.NoiseModel(1e-3, 1e-3, decoherence=C.Decoherence(1e-4, schedule="lines")))]
    samplers = [tmcs.Sampler(c) for c in circs]
    shots = 64 * 16
    outs = [s.alloc(shots) for s in samplers]
    jobs = [(s.handle, shots, 7, d, o) for s, (d, o) in zip(samplers, outs)]
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def best(batches):
        times = []
        for _ in range(23):
            a.record()
            for x in batches:
                tmcs.tmcs_batch_sample(x)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times[3:])

    alone = best([[j] for j in jobs])
    together = best([jobs])
    tmcs.tmcs_check_device()
    # one after the other: the same as alone; side by side: near a third
    assert together < 0.75 * alone, (together, alone)
    for s in samplers:
        s.close()
