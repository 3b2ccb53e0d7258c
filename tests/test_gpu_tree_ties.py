"""The best-first tree of up to 32 nodes on lists with exact ties: the loop that takes a row's entries in
order hands over to the loop on entry masks at the first tie among a node's children, and the 32nd node
takes the anchor's lane.  Identical rows of W_lm give identical logits, so every position's list holds
runs of equal values; the selection is compared with the definition computed the slow way from the
lists that the step itself returns, exactly."""
import numpy as np
import pytest
import torch

from paper_2605_29707_gb300 import inputs
from paper_2605_29707_gb300.step import DraftStep

pytestmark = pytest.mark.gpu


def _tree(ids, logp, N):
    """Pops of greatest (score, lower token, lower parent index), scores summed in fp32."""
    K, k = ids.shape
    front = [(np.float32(0.0) + logp[0, j], int(ids[0, j]), -1, 1) for j in range(k)]
    out = []
    while len(out) < N and front:
        best = min(range(len(front)), key=lambda i: (-front[i][0], front[i][1], front[i][2]))
        s, t, par, d = front.pop(best)
        if d < K:
            front += [(np.float32(s + logp[d, j]), int(ids[d, j]), len(out), d + 1) for j in range(k)]
        out.append((par, t, d, s))
    return out


@pytest.mark.parametrize("repeat", [1, 2, 5], ids=["distinct", "pairs", "fives"])
@pytest.mark.parametrize("K,k,N", [(4, 4, 8), (6, 8, 31), (6, 8, 32), (1, 8, 8), (3, 16, 32), (5, 3, 32)])
def test_tree_is_the_definition_on_the_returned_lists(K, k, N, repeat):
    B, H, V = 3, 64, 1200
    cfg = inputs.custom_config("ties", B=B, K=K, H=H, V=V, Ds=32, R=16, k=k, N=N, seed=11 + repeat, hidden_kind="rms1")
    wl = inputs.make_workload(cfg)
    w = dict(wl.weights)
    w["w_lm"] = np.repeat(w["w_lm"][: V // repeat], repeat, axis=0)
    w["w2"] = np.repeat(w["w2"][: V // repeat], repeat, axis=0)
    st = DraftStep(w, B, K, H, V, k, N, Ds=32, R=16, device="cuda:0")
    out = st.run(torch.from_numpy(wl.hidden.view(np.int16)).view(torch.bfloat16).cuda(),
                 torch.from_numpy(wl.prefix_ids).cuda())
    for b in range(B):
        ref = _tree(out["topk_ids"][b], out["topk_logp"][b], N)
        got = list(zip(out["tree_parent"][b], out["tree_token"][b], out["tree_depth"][b], out["tree_score"][b]))
        assert [tuple(map(int, r[:3])) for r in got] == [r[:3] for r in ref]
        assert all(np.float32(g[3]) == r[3] for g, r in zip(got, ref))
