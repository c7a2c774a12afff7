"""The gap count of the frame, barrier and pipelined kernels against its
definition.

They have their own form of the one-read count (rounded by a float-to-int
conversion; the decoupled kernel's walkers round by an addition), so it is
compared at every table boundary too, on the words of test_gpu_gap.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2504_05611_gb300 import tmcs  # noqa: E402
from test_gpu_gap import PROBS, boundary_words, expected_counts  # noqa: E402


@pytest.mark.parametrize("p", PROBS)
def test_counts_match_definition(p):
    table = oracle.gap_table(p)
    words = boundary_words(table, np.random.default_rng(int(p * 1e9) + 4))
    dw = torch.from_numpy(words.view(np.int32)).cuda()
    got = tmcs.tmcs_debug_gap_counts(p, dw, 4).cpu().numpy()
    assert np.array_equal(got, expected_counts(table, words))


def test_other_methods_are_refused():
    dw = torch.zeros(4, dtype=torch.int32, device="cuda")
    for method in (-1, 3, 5):
        with pytest.raises(tmcs.TmcsError):
            tmcs.tmcs_debug_gap_counts(0.1, dw, method)
