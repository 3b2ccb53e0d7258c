"""Rows of W2 that hold an infinite weight, in the sequential loop's tensor-core phase C: u's terms after the
first have either sign, and their products with the weight must not turn the row's logit, infinite of
u's sign, into NaN.  Column 0 of every third row is -inf where u_0 > 0 at every step (b1 is 8 there), so
that those tokens have no probability and every other one keeps its own; rows of the resident blocks and
of the rest, against the oracle by the teacher-forced rules of tests/test_gpu_rollout.py."""
import dataclasses

import numpy as np
import pytest

from paper_2605_29707_gb300 import inputs
from tests.test_gpu_rollout import _check, _check_gumbel, _full_emb, _run_gpu

pytestmark = pytest.mark.gpu

MINUS_INF, EIGHT = 0xFF80, 0x4100  # bf16


@pytest.mark.parametrize("table", [False, True], ids=["project", "table"])
@pytest.mark.parametrize("B,R,rows", [(1, 256, 6 * 128 + 150), (4, 64, 40), (4, 256, 5 * 128 + 150), (8, 256, 4 * 128 + 20)])
def test_infinite_weights_match_oracle(B, R, rows, table):
    cfg = inputs.custom_config("loop-inf", B=B, K=3, H=64, V=152 * rows, Ds=32, R=R, seed=95, biases=True)
    wl = _full_emb(inputs.make_workload(cfg))
    w = {n: a.copy() if n in ("w2", "b1") else a for n, a in wl.weights.items()}
    w["w2"][::3, 0] = MINUS_INF
    w["b1"][0] = EIGHT
    wl = dataclasses.replace(wl, weights=w)
    tokens, logp = _run_gpu(wl, table=table)
    assert (tokens % 3 != 0).all() and np.isfinite(logp).all()
    _check(wl, table=table)
    _check_gumbel(wl, seed=92, table=table)
