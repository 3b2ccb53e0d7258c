"""Batches of 33 to 128 positions: the vocabulary GEMM's W_lm segment streams beside the GRU on 64- and
128-column accumulator blocks, fewer than the tiles of a CTA, so that blocks are used again; u comes
from 4 x 4 tiles of (rank row, position).  Against the oracle by tests/test_gpu_parity.py's rules."""
import pytest

from paper_2605_29707_gb300 import inputs
from tests.test_gpu_parity import _check, _run_gpu

pytestmark = pytest.mark.gpu

# M at the edges of the two block widths and of a position tile; V past 152 x 128 x 4 rows (five tiles
# a CTA over four 128-column blocks), ragged; the three list lengths; d_s past one 1024-column slice
CASES = {
    "m33": dict(B=3, K=11, H=64, V=152 * 128 * 2 + 5, Ds=64, R=64, k=8, N=16, seed=81),
    "m64-k10": dict(B=4, K=16, H=128, V=152 * 128 * 3 - 3, Ds=136, R=72, k=10, N=32, seed=82, biases=True),
    "m65": dict(B=5, K=13, H=64, V=152 * 128 * 4 + 100, Ds=64, R=64, k=8, N=9, seed=83),
    "m128-k20": dict(B=8, K=16, H=64, V=152 * 128 * 4 + 1, Ds=256, R=40, k=20, N=24, seed=84, biases=True),
    # 100 sequences of one position on a small d_s: two gate evaluations a thread beside the vocabulary GEMM
    "m100-b100": dict(B=100, K=1, H=64, V=3001, Ds=64, R=64, k=4, N=4, seed=86),
    "m120-b40": dict(B=40, K=3, H=64, V=3001, Ds=64, R=64, k=4, N=8, seed=87, biases=True),
    "m102-ds1032": dict(B=6, K=17, H=64, V=3001, Ds=1032, R=64, k=4, N=12, seed=85),
}


@pytest.mark.parametrize("table", [False, True], ids=["project", "table"])
@pytest.mark.parametrize("name", list(CASES))
def test_overlapped_batches_match_oracle(name, table):
    cfg = inputs.custom_config(name, **CASES[name])
    wl = inputs.make_workload(cfg)
    _, out, _, _ = _run_gpu(wl, table=table)
    ex_topk, ex_tree = _check(wl, out)
    assert ex_topk <= max(1, cfg.M * cfg.k // 50)
    assert ex_tree <= max(1, cfg.B * cfg.N // 10)
