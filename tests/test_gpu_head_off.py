"""Up to 128 positions without the correction branch: the vocabulary GEMM alone on the SMs, which transposes a
whole 128-row tile at a time.  Vocabularies that end in the middle of a tile, of a warp's rows and of an
epilogue thread's chunk, one to three tiles a CTA (152 SMs), the four accumulator widths, each list length,
with and without b2, against the oracle."""
import pytest

from paper_2605_29707_gb300 import inputs
from tests.test_gpu_parity import _check, _run_gpu

pytestmark = pytest.mark.gpu

SHAPES = [(1, 13, 152 * 128 + 1, 8, False), (2, 16, 3001, 20, True), (4, 16, 152 * 128 * 2 + 65, 10, False),
          (5, 12, 152 * 128 - 31, 17, True), (5, 13, 152 * 128 * 2 + 33, 8, True), (8, 16, 152 * 128 + 127, 16, False),
          (8, 16, 97, 32, True)]


@pytest.mark.parametrize("B,K,V,k,biases", SHAPES)
def test_head_off_matches_oracle(B, K, V, k, biases):
    cfg = inputs.custom_config("off", B=B, K=K, H=200, V=V, Ds=64, R=64, k=k, N=6, seed=V % 89, biases=biases)
    wl = inputs.make_workload(cfg)
    _, out, _, _ = _run_gpu(wl, head_on=False)
    ex_topk, ex_tree = _check(wl, out, head_on=False)
    assert ex_topk <= max(1, cfg.M * cfg.k // 50)
    assert ex_tree <= max(1, cfg.B * cfg.N // 10)
