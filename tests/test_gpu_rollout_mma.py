"""The sequential loop's phase C on the tensor cores beyond two sequences and without the input
table: u's three bf16 terms, accumulators of 16 and 32 columns, and 16-row tiles of the rows past
the resident blocks, at their edges, against the oracle by the teacher-forced rules and tolerances of
tests/test_gpu_rollout.py."""
import pytest

from paper_2605_29707_gb300 import inputs
from tests.test_gpu_rollout import _check, _check_gumbel, _full_emb

pytestmark = pytest.mark.gpu

# Rows a CTA keeps past its resident 128-row blocks (152 SMs, r = 256: 4 blocks at B = 5..8, 5 at
# B = 3 and 4, 6 at B <= 2): none, one, a ragged tile, just past one tile of each of the eight warps.
CASES = [
    inputs.custom_config("loop-mma-b8-blocks", B=8, K=3, H=64, V=152 * 512, Ds=32, R=256, seed=71),
    inputs.custom_config("loop-mma-b8-one", B=8, K=3, H=64, V=152 * 512 + 1, Ds=32, R=256, seed=72, biases=True),
    inputs.custom_config("loop-mma-b5", B=5, K=3, H=64, V=152 * 531 - 3, Ds=264, R=256, seed=73),
    inputs.custom_config("loop-mma-b4", B=4, K=3, H=64, V=152 * (640 + 129) - 7, Ds=32, R=256, seed=74, biases=True),
    inputs.custom_config("loop-mma-b3-r64", B=3, K=4, H=64, V=152 * 40 + 5, Ds=64, R=64, seed=75),
    inputs.custom_config("loop-mma-b2", B=2, K=3, H=64, V=152 * (768 + 17), Ds=32, R=256, seed=76),
    inputs.custom_config("loop-mma-b1-r192", B=1, K=3, H=64, V=152 * 1300 + 11, Ds=32, R=192, seed=77, biases=True),
]


@pytest.mark.parametrize("table", [False, True], ids=["project", "table"])
@pytest.mark.parametrize("cfg", CASES, ids=[c.name for c in CASES])
def test_loop_tensor_core_rows_match_oracle(cfg, table):
    wl = _full_emb(inputs.make_workload(cfg))
    _check(wl, table=table)
    _check_gumbel(wl, seed=91, table=table)
