"""A staging copy of the row draw (domino_verify_tree_sample) that never lands: the wait for it runs out,
the row is read directly, and every output is what it is without the hook.  Nothing traps or hangs."""
import time

import numpy as np
import pytest

from paper_2605_29707_gb300 import binding, inputs
from tests import test_gpu_verify_sample as sample

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [12, 4096, 20000])  # slices of one chunk (and empty ones), and of four
def test_withheld_copy_changes_no_draw(V):
    B, N, row = 2, 4, 6  # row 1 of sequence 1
    case = inputs.make_verify_case(B, N, V, 51, p_plant=0.9, chain=True, margin=5.0)
    u = sample._uniforms(B, N, 51)
    want = sample._run_gpu(case, u, 1.0)
    assert binding.domino_debug_hold(binding.DOMINO_HOLD_ROW_COPY, row) == 0
    t0 = time.perf_counter()
    try:
        got = sample._run_gpu(case, u, 1.0)
    finally:
        assert binding.domino_debug_hold(binding.DOMINO_HOLD_OFF) == 0
    assert 0.5 < time.perf_counter() - t0 < 30.0  # the wait did run out
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a, b)
    sample._check(case, u, 1.0)  # the hook held one launch only
