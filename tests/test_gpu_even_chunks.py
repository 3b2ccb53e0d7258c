"""Equal vocabulary chunks: a CTA's last tile is shorter than 128 rows, with tensor maps of its own, in
the block step of 33 to 128 positions (whole tiles at fewer).  Vocabularies that put 8, 120 and 128 rows
into the last tile (152 SMs), ragged, against the oracle; and a workspace that only holds the records of
whole-tile chunks, which a step still accepts."""
import numpy as np
import pytest
import torch

from paper_2605_29707_gb300 import binding, inputs
from paper_2605_29707_gb300.step import DraftStep
from tests.test_gpu_parity import _check, _run_gpu

pytestmark = pytest.mark.gpu

SHAPES = [(1, 5, 152 * 136 - 3, 6), (2, 9, 152 * 248 + 1 - 152 * 8, 12), (3, 11, 152 * 136 - 3, 6),
          (4, 16, 152 * 248 + 1 - 152 * 8, 12), (5, 13, 152 * 256, 8),
          (5, 13, 152 * 248 + 1 - 152 * 8, 12), (8, 16, 152 * 264 - 700, 8)]


@pytest.mark.parametrize("B,K,V,k", SHAPES)
def test_short_last_tiles_match_oracle(B, K, V, k):
    cfg = inputs.custom_config("even", B=B, K=K, H=72, V=V, Ds=64, R=72, k=k, N=5, seed=V % 97, biases=True)
    wl = inputs.make_workload(cfg)
    _, out, _, _ = _run_gpu(wl)
    _check(wl, out)


def test_a_workspace_of_whole_tile_chunks_is_accepted():
    B, K, V, k = 3, 11, 152 * 129, 8  # 129 rows a CTA: 143 equal chunks, 77 of two whole tiles
    cfg = inputs.custom_config("even-ws", B=B, K=K, H=64, V=V, Ds=64, R=64, k=k, N=5, seed=5)
    wl = inputs.make_workload(cfg)
    st = DraftStep(wl.weights, B, K, cfg.H, V, k, 5, Ds=64, R=64, device="cuda:0")
    records = B * K * (2 + 2 * 8) * 4
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = -(-(-(-V // sms)) // 8) * 8
    equal, whole = -(-V // rows), -(-(-(-V // 128)) // 2)
    st.ws_bytes -= records * (equal - whole) // 256 * 256
    hidden = torch.from_numpy(wl.hidden.view(np.int16)).view(torch.bfloat16).cuda()
    ids = torch.from_numpy(wl.prefix_ids).cuda()
    _check(wl, st.run(hidden, ids))
    st.ws_bytes -= records * whole
    assert st.enqueue(hidden, ids) == binding.DOMINO_ERR_INVALID_ARG
