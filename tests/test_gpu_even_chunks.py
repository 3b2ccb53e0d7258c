"""Equal vocabulary chunks: a CTA's last tile is shorter than 128 rows, with tensor maps of its own, in
the block step up to 128 positions, where the vocabulary stream outlasts the GRU (and whole tiles where it
does not).  Vocabularies that put 8, 120 and 128 rows into the last tile (152 SMs), ragged, against the
oracle; and a workspace that only holds the records of whole-tile chunks, which a step still accepts."""
import numpy as np
import pytest
import torch

from paper_2605_29707_gb300 import binding, inputs
from paper_2605_29707_gb300.step import DraftStep
from tests.test_gpu_parity import _check, _run_gpu

pytestmark = pytest.mark.gpu

SHAPES = [(1, 5, 152 * 136 - 3, 6), (2, 9, 152 * 248 + 1 - 152 * 8, 12), (4, 16, 152 * 256, 8), (8, 16, 152 * 264 - 700, 8)]


# H wide enough that the stream outlasts the GRU on each position block (16, 32, 64 and 128 columns)
LONG = [(1, 2, 152 * 136 - 3, 6, 1920), (12, 2, 152 * 264 - 700, 8, 2112), (40, 1, 152 * 248 - 1208, 12, 3264),
        (72, 1, 152 * 264 - 700, 8, 3072)]


@pytest.mark.parametrize("B,K,V,k", SHAPES)
def test_whole_tiles_of_short_streams_match_oracle(B, K, V, k):
    cfg = inputs.custom_config("even", B=B, K=K, H=72, V=V, Ds=64, R=72, k=k, N=5, seed=V % 97, biases=True)
    wl = inputs.make_workload(cfg)
    _, out, _, _ = _run_gpu(wl)
    _check(wl, out)


@pytest.mark.parametrize("B,K,V,k,H", LONG)
def test_short_last_tiles_match_oracle(B, K, V, k, H):
    cfg = inputs.custom_config("even-long", B=B, K=K, H=H, V=V, Ds=64, R=72, k=k, N=K, seed=V % 97, biases=True)
    wl = inputs.make_workload(cfg)
    _, out, _, _ = _run_gpu(wl)
    _check(wl, out)


@pytest.mark.parametrize("head_on", [True, False])
def test_a_workspace_of_whole_tile_chunks_is_accepted(head_on):
    B, K, V, k = 2, 2, 152 * 129, 8  # 129 rows a CTA: 143 equal chunks, 77 of two whole tiles
    cfg = inputs.custom_config("even-ws", B=B, K=K, H=2176, V=V, Ds=64, R=64, k=k, N=5, seed=5)
    wl = inputs.make_workload(cfg)
    st = DraftStep(wl.weights, B, K, cfg.H, V, k, 5, Ds=64, R=64, device="cuda:0", head_on=head_on)
    records = B * K * (2 + 2 * 8) * 4
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = -(-(-(-V // sms)) // 8) * 8
    equal, whole = -(-V // rows), -(-(-(-V // 128)) // 2)
    st.ws_bytes -= records * (equal - whole) // 256 * 256
    hidden = torch.from_numpy(wl.hidden.view(np.int16)).view(torch.bfloat16).cuda()
    ids = torch.from_numpy(wl.prefix_ids).cuda()
    _check(wl, st.run(hidden, ids), head_on=head_on)
    st.ws_bytes -= records * whole
    assert st.enqueue(hidden, ids) == binding.DOMINO_ERR_INVALID_ARG
