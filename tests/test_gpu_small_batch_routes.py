"""Routes of a block step of 33 to 128 positions that the other tests' sizes do not take, against the oracle by
tests/test_gpu_parity.py's rules.

The GRU that takes the whole SM at a d_s of 512 and more (9 and more sequences): packed states read by the
in-kernel u, and input-gate sums from four to ten split-K partial sums (three are held, or six; the rest
are added one by one), with one and two gate evaluations a thread.  The GRU that computes its own
projections over more than 32 positions (a small r): three to eight tiles of 16 positions.  The host
entry point with a workspace that holds the records of whole-tile vocabulary chunks only."""
import numpy as np
import pytest
import torch

from paper_2605_29707_gb300 import binding, inputs
from paper_2605_29707_gb300.step import DraftStep
from tests.test_gpu_parity import _check, _run_gpu

pytestmark = pytest.mark.gpu

CASES = {
    "wide-6-splits": dict(B=12, K=8, H=768, V=3001, Ds=1024, R=64, k=8, N=12, seed=101),
    "wide-k20": dict(B=9, K=13, H=400, V=3001, Ds=1024, R=72, k=20, N=16, seed=102, biases=True),
    "wide-ds1032": dict(B=16, K=4, H=320, V=3001, Ds=1032, R=64, k=8, N=9, seed=103),
    "wide-7-splits": dict(B=32, K=4, H=832, V=3001, Ds=512, R=64, k=4, N=6, seed=104, biases=True),
    "wide-two-evaluations": dict(B=40, K=3, H=640, V=3001, Ds=512, R=40, k=4, N=6, seed=105),
    "fused-m48": dict(B=3, K=16, H=256, V=3001, Ds=1024, R=64, k=8, N=16, seed=106, biases=True),
    "fused-m128": dict(B=8, K=16, H=200, V=3001, Ds=1024, R=32, k=12, N=16, seed=107),
    "fused-k64": dict(B=1, K=64, H=264, V=152 * 128 + 5, Ds=256, R=16, k=4, N=40, seed=108),
}
LAUNCHES = {"wide": 6, "fused": 3}  # without a table


@pytest.mark.parametrize("table", [False, True], ids=["project", "table"])
@pytest.mark.parametrize("name", list(CASES))
def test_routes_match_oracle(name, table):
    cfg = inputs.custom_config(name, **CASES[name])
    n = binding.domino_launches_per_step(cfg.B, cfg.K, cfg.H, cfg.V, cfg.Ds, cfg.R, cfg.k, cfg.N)
    assert n == LAUNCHES[name.split("-")[0]]
    wl = inputs.make_workload(cfg)
    _, out, _, _ = _run_gpu(wl, table=table)
    ex_topk, ex_tree = _check(wl, out)
    assert ex_topk <= max(1, cfg.M * cfg.k // 50)
    assert ex_tree <= max(1, cfg.B * cfg.N // 10)


def test_host_entry_accepts_a_workspace_of_whole_tile_chunks():
    """129 rows a CTA: 145 equal chunks, 77 of two whole tiles.  Three calls with the smaller size (the third
    replays a graph), then one with the full size on the same buffers, each against the oracle."""
    B, K, V, k = 3, 11, 152 * 129, 8
    cfg = inputs.custom_config("even-ws-host", B=B, K=K, H=64, V=V, Ds=64, R=64, k=k, N=5, seed=6)
    wl = inputs.make_workload(cfg)
    st = DraftStep(wl.weights, B, K, cfg.H, V, k, 5, Ds=64, R=64, device="cuda:0")
    hidden = torch.from_numpy(wl.hidden.view(np.int16)).pin_memory()
    ids = torch.from_numpy(wl.prefix_ids).pin_memory()
    new = lambda shape, dt: torch.empty(shape, dtype=dt).pin_memory()  # noqa: E731
    out = {"topk_ids": new((B, K, k), torch.int32), "topk_logp": new((B, K, k), torch.float32),
           "tree_parent": new((B, 5), torch.int32), "tree_token": new((B, 5), torch.int32),
           "tree_depth": new((B, 5), torch.int32), "tree_score": new((B, 5), torch.float32)}

    def call():
        for t in out.values():
            t.fill_(-7)
        rc = st.run_host(hidden, ids, out)
        if rc == 0:
            _check(wl, {n: t.numpy() for n, t in out.items()})
        return rc

    full = st.ws_host_bytes
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    records = B * K * (2 + 2 * 8) * 4
    rows = -(-(-(-V // sms)) // 8) * 8
    equal, whole = -(-V // rows), -(-(-(-V // 128)) // 2)
    st.ws_host_bytes = full - records * (equal - whole) // 256 * 256
    assert [call() for _ in range(3)] == [0, 0, 0]
    st.ws_host_bytes = full
    assert call() == 0
    st.ws_host_bytes = full - records * equal
    assert call() == binding.DOMINO_ERR_INVALID_ARG
