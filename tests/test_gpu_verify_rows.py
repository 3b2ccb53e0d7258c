"""Tree verification of more rows than the chip has SMs: the argmax takes two CTAs a row, and the row
draw asks for later rows ahead of time.  Small vocabularies put the slice ends where they can go wrong
(empty and ragged slices, scalar and vector loads); the rules are those of tests/test_gpu_verify.py and
tests/test_gpu_verify_sample.py."""
import numpy as np
import pytest

from paper_2605_29707_gb300 import inputs
from tests import test_gpu_verify as greedy
from tests import test_gpu_verify_sample as sample

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [4, 7, 1000, 1003, 20000])
def test_many_rows_match_oracle(V):
    B, N = 20, 8  # 180 rows
    # (a chain below 1000 ids: siblings carry distinct tokens)
    case = inputs.make_verify_case(B, N, V, 41 + V, p_plant=0.8, chain=V < 1000, margin=9.0)
    # the same maximum twice in some rows, once on either side of the half: the lower id
    case.target[3, :, V // 2 - 1] = case.target[3, :, V - 1] = 60.0
    greedy._check(case)
    case.target[3] = np.minimum(case.target[3], 20.0)
    sample._check(case, sample._uniforms(B, N, 5), 1.0)
