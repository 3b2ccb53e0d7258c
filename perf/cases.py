"""The work that a speculative-decoding server has this library do, as cases that can be timed.

A serving loop alternates two calls: draft a block for every running sequence (the block step
`DraftStep`, or the sequential draft loop `domino_rollout_*` when the prefix tokens are not known
yet) and verify the drafted trees against the target's logits (`domino_verify_tree_*`).  The sizes
are those of the repository's configurations (hidden widths 2048, 4096 and 5120, a vocabulary of
151936, d_s = 1024, r = 256, blocks of 16, batches of 1 to 64) with ragged batches and blocks among
them.  Weights are random-init of that shape; the hidden states are scaled so that the base
distribution has about 3 nats of entropy, as a trained head's has.
"""
import heapq
import math

import torch

from paper_2605_29707_gb300 import binding
from paper_2605_29707_gb300.step import DraftStep

DS, R = 1024, 256
VOCAB = 151936
WSTD = 0.02
LOGIT_STD = 5.1  # of the base logits: about 3 nats of entropy over 151936 ids


# ------------------------------------------------------------------------------------- cases
def _step(name, B, K, H, V=VOCAB, k=8, N=16, table=False, biases=False, head=True, host=False):
    return dict(name=name, kind="step", B=B, K=K, H=H, V=V, k=k, N=N, table=table, biases=biases, head=head, host=host)


def _rollout(name, rule, B, K, H, V=VOCAB, table=True, biases=False):
    return dict(name=name, kind="rollout", rule=rule, B=B, K=K, H=H, V=V, table=table, biases=biases)


def _verify(name, rule, B, N, V=VOCAB):
    return dict(name=name, kind="verify", rule=rule, B=B, N=N, V=V)


def listed():
    return [
        # one interactive sequence: the smallest call, checking one drafted tree at temperature 0
        _verify("verify-greedy-b1", "greedy", B=1, N=16),
        # a serving batch's trees checked at temperature 1, where the logits are far larger than L2
        _verify("verify-sample-b32", "sample", B=32, N=16),
        # one sequence on a small target, called from a host program with its buffers in host memory
        _step("step-h2048-b1-host", B=1, K=16, H=2048, host=True),
        # one sequence on a mid-size target: the latency that the paper quotes
        _step("step-h4096-b1", B=1, K=16, H=4096),
        # a few concurrent users
        _step("step-h4096-b4", B=4, K=16, H=4096),
        # an uneven batch with the paper's block of 15 drafted tokens, and a head that has biases
        _step("step-h4096-b7-k15", B=7, K=15, H=4096, biases=True),
        # a batch between the tuned ones, on a server that keeps the input-projection table
        _step("step-h4096-b20-table", B=20, K=16, H=4096, table=True),
        # a serving batch on a mid-size target
        _step("step-h4096-b32", B=32, K=16, H=4096),
        # the largest: a full serving batch on a large target, wider lists and a larger tree
        _step("step-h5120-b64", B=64, K=16, H=5120, k=10, N=32),
        # one sequence drafted token by token at temperature 0, with the table
        _rollout("loop-greedy-h4096-b1", "greedy", B=1, K=16, H=4096),
        # a few users drafted token by token, sampled by the seeded race
        _rollout("loop-race-h4096-b4", "race", B=4, K=16, H=4096),
        # two users on a small target without room for the table, sampled by the caller's uniforms
        _rollout("loop-cdf-h2048-b2-notable", "cdf", B=2, K=16, H=2048, table=False),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(("step", "rollout", "verify"), (6, 3, 2))[0]
    V = rng.choice((VOCAB, VOCAB, _log_int(rng, 32000, VOCAB)))
    if kind == "step":
        B, K = _log_int(rng, 1, 64), rng.choice((16, 16, 15, rng.randint(4, 16)))
        c = _step("", B, K, rng.choice((2048, 4096, 5120)), V, k=rng.choice((4, 8, 8, 10)), N=rng.randint(8, 32),
                  table=rng.random() < 0.4, biases=rng.random() < 0.3, head=rng.random() < 0.9, host=B <= 2 and rng.random() < 0.3)
    elif kind == "rollout":
        c = _rollout("", rng.choice(("greedy", "race", "cdf")), _log_int(rng, 1, 8), rng.choice((16, rng.randint(4, 16))),
                     rng.choice((2048, 4096)), V, table=rng.random() < 0.6, biases=rng.random() < 0.3)
    else:
        c = _verify("", rng.choice(("greedy", "sample")), _log_int(rng, 1, 64), rng.randint(8, 32), V)
    del c["name"]
    return c


# ------------------------------------------------------------------------------------ inputs
def _gen(seed, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 64 + n)
    return g


def _normal(shape, std, g, dtype=torch.bfloat16):
    out = torch.empty(shape, dtype=dtype, device="cuda")
    rows = max(1, (1 << 26) // max(1, math.prod(shape[1:])))
    for a in range(0, shape[0], rows):  # in pieces: the fp32 draws of a whole matrix would be large
        b = min(shape[0], a + rows)
        out[a:b] = torch.randn((b - a, *shape[1:]), generator=g, device="cuda").mul_(std)
    return out


def _weights(c, seed):
    H, V, head = c["H"], c["V"], c.get("head", True)
    shapes = {"w_lm": (V, H)}
    if head:
        shapes.update(emb=(V, H), w_ih=(3 * DS, H), w_hh=(3 * DS, DS), w1=(R, H + DS), w2=(V, R))
    w = {n: _normal(s, WSTD, _gen(seed, i)) for i, (n, s) in enumerate(shapes.items())}
    if c["biases"]:
        sizes = {"b2": (V,)}
        if head:
            sizes.update(b_ih=(3 * DS,), b_hh=(3 * DS,), b1=(R,))
        w.update({n: _normal(s, 0.1, _gen(seed, 16 + i)) for i, (n, s) in enumerate(sizes.items())})
    return w


def _hidden(c, seed):
    return _normal((c["B"], c["K"], c["H"]), LOGIT_STD / (WSTD * math.sqrt(c["H"])), _gen(seed, 32))


def _ids(shape, V, seed):
    return torch.randint(0, V, shape, generator=_gen(seed, 33), device="cuda", dtype=torch.int32)


def _verify_inputs(c, seed):
    """Random trees (parents before children) and the target's logits: after seven nodes of ten one child's token is
    likely (raised above the row's maximum), as after a draft that the target mostly agrees with."""
    B, N, V = c["B"], c["N"], c["V"]
    g = torch.Generator().manual_seed(int(seed) * 64 + 40)
    parent = torch.stack([torch.stack([torch.randint(-1, max(1, i), (), generator=g) if i else torch.tensor(-1)
                                       for i in range(N)]) for _ in range(B)])
    token = torch.randint(0, V, (B, N), generator=g)
    keep = torch.rand(B, N, generator=g) < 0.7
    target = _normal((B * (N + 1), V), LOGIT_STD, _gen(seed, 41), torch.float32).view(B, N + 1, V)
    top = target.amax(-1).cpu()
    bb, ii = torch.nonzero(keep, as_tuple=True)
    rows = parent[bb, ii] + 1
    target[bb.cuda(), rows.cuda(), token[bb, ii].cuda()] = (top[bb, rows] + 2.0 + 0.01 * ii).cuda()
    uni = torch.rand(B, N + 1, generator=_gen(seed, 42), device="cuda")
    return parent.int().cuda().contiguous(), token.int().cuda().contiguous(), target, uni


def prepare(case, seed):
    c = case
    if c["kind"] == "verify":
        parent, token, target, uni = _verify_inputs(c, seed)
        B, N = c["B"], c["N"]
        new = lambda *s: torch.empty(s, dtype=torch.int32, device="cuda")  # noqa: E731
        return dict(c=c, parent=parent, token=token, target=target, uni=uni,
                    out=dict(row=new(B, N + 1), nodes=new(B, N), count=new(B), bonus=new(B)))
    w = _weights(c, seed)
    if c["kind"] == "step":
        st = DraftStep(w, c["B"], c["K"], c["H"], c["V"], c["k"], c["N"], Ds=DS, R=R, head_on=c["head"],
                       input_table=c["table"])
        hidden, ids = _hidden(c, seed), _ids((c["B"], c["K"]), c["V"], seed)
        if not c["host"]:
            return dict(c=c, step=st, hidden=hidden, ids=ids)
        out = {n: torch.empty(t.shape, dtype=t.dtype).pin_memory() for n, t in _outputs(c, st).items()}
        return dict(c=c, step=st, hidden=hidden.cpu().pin_memory(), ids=ids.cpu().pin_memory(), out=out)
    B, K, H, V = c["B"], c["K"], c["H"], c["V"]
    table = None
    if c["table"]:
        table = torch.empty(binding.domino_input_table_bytes(V, DS) // 4, dtype=torch.float32, device="cuda")
        _ok(binding.domino_build_input_table(w["emb"], w["w_ih"], V, H, DS, table, torch.cuda.current_stream()))
    head = binding.make_head(**{n: w.get(n) for n in ("emb", "w_ih", "w_hh", "b_ih", "b_hh", "w1", "b1", "w2", "b2")},
                             Ds=DS, R=R, x_table=table)
    nb = binding.domino_rollout_workspace_bytes(B, K, H, V, DS, R)
    return dict(c=c, w=w, table=table, head=head, hidden=_hidden(c, seed), anchors=_ids((B,), V, seed),
                uni=torch.rand(B, K, generator=_gen(seed, 34), device="cuda"), key=int(seed) * 7919 + 1,
                ws=torch.zeros(nb, dtype=torch.uint8, device="cuda"), nb=nb,
                out=dict(tokens=torch.empty(B, K, dtype=torch.int32, device="cuda"),
                         logp=torch.empty(B, K, dtype=torch.float32, device="cuda")))


def _ok(rc):
    if rc != 0:
        raise binding.DominoError(rc)


def _outputs(c, st):
    B, K, k, N = c["B"], c["K"], c["k"], c["N"]
    return dict(topk_ids=st.topk_ids.view(B, K, k), topk_logp=st.topk_logp.view(B, K, k),
                tree_parent=st.tree_parent.view(B, N), tree_token=st.tree_token.view(B, N),
                tree_depth=st.tree_depth.view(B, N), tree_score=st.tree_score.view(B, N))


def run(state):
    s, c = state, state["c"]
    if c["kind"] == "step":
        st = s["step"]
        if c["host"]:
            _ok(st.run_host(s["hidden"], s["ids"], s["out"]))
            return s["out"]
        _ok(st.enqueue(s["hidden"], s["ids"]))
        return _outputs(c, st)
    o, stream = s["out"], torch.cuda.current_stream()
    if c["kind"] == "verify":
        if c["rule"] == "greedy":
            rc = binding.domino_verify_tree_greedy(s["target"], s["parent"], s["token"], c["B"], c["N"], c["V"], o["row"],
                                                   o["nodes"], o["count"], o["bonus"], stream)
        else:
            rc = binding.domino_verify_tree_sample(s["target"], s["parent"], s["token"], s["uni"], 1.0, c["B"], c["N"],
                                                   c["V"], o["row"], o["nodes"], o["count"], o["bonus"], stream)
        _ok(rc)
        return o
    args = (s["w"]["w_lm"], s["head"], c["B"], c["K"], c["H"], c["V"], o["tokens"], o["logp"], s["ws"], s["nb"], stream)
    if c["rule"] == "greedy":
        rc = binding.domino_rollout_greedy(s["hidden"], s["anchors"], *args)
    elif c["rule"] == "race":
        rc = binding.domino_rollout_sample_gumbel(s["hidden"], s["anchors"], s["key"], *args)
    else:
        rc = binding.domino_rollout_sample(s["hidden"], s["anchors"], s["uni"], *args)
    _ok(rc)
    return o


def work(case):
    c = case
    if c["kind"] == "verify":
        rows = c["B"] * (c["N"] + 1)
        return {"bytes": rows * c["V"] * 4 + c["B"] * c["N"] * 12 + rows * 8, "flops": 2 * rows * c["V"]}
    B, K, H, V = c["B"], c["K"], c["H"], c["V"]
    M, head = B * K, c.get("head", True)
    nbytes, flops = V * H * 2 + M * H * 2 + M * 4, 2 * M * V * H
    if head:
        nbytes += (V * R + R * (H + DS) + 3 * DS * DS) * 2
        flops += 2 * M * (V * R + R * (H + DS) + 3 * DS * DS)
        if c["table"]:
            nbytes += M * 3 * DS * 4
        else:
            nbytes += M * H * 2 + 3 * DS * H * 2
            flops += 2 * M * 3 * DS * H
    if c["biases"]:
        nbytes += V * 2 + ((6 * DS + R) * 2 if head else 0)
    nbytes += M * c["k"] * 8 + B * c["N"] * 16 if c["kind"] == "step" else M * 8
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------- the same in 64 bits
def _bias(w, n):
    return w[n].double() if n in w else 0.0


def _gru_step(w, h, ids):
    """One step of torch.nn.GRU on the embeddings of `ids` [B], from h [B, DS]."""
    x = w["emb"][ids.long()].double() @ w["w_ih"].double().T + _bias(w, "b_ih")
    a = h @ w["w_hh"].double().T + _bias(w, "b_hh")
    xr, xz, xn = x.split(DS, -1)
    hr, hz, hn = a.split(DS, -1)
    r, z = torch.sigmoid(xr + hr), torch.sigmoid(xz + hz)
    return (1 - z) * torch.tanh(xn + r * hn) + z * h


def _code(w, hid, S):
    v = torch.cat((hid, S), -1) @ w["w1"].double().T + _bias(w, "b1")
    return v * torch.sigmoid(v)


def _logits(w, hid, u):
    """hid [M, H], u [M, R] or None -> [M, V]."""
    out = torch.empty(hid.shape[0], w["w_lm"].shape[0], dtype=torch.float64, device="cuda")
    for a in range(0, out.shape[1], 16384):
        b = min(out.shape[1], a + 16384)
        out[:, a:b] = hid @ w["w_lm"][a:b].double().T
        if u is not None:
            out[:, a:b] += u @ w["w2"][a:b].double().T
    return out + _bias(w, "b2")


def _tree_scores(ids, logp, N):
    """Cumulative log-probabilities of the N best nodes, best first (ids and logp [K, k])."""
    K = len(ids)
    heap = [(-s, t, -1, 1) for s, t in zip(logp[0], ids[0])]
    heapq.heapify(heap)
    scores = []
    while len(scores) < N:
        s, _, _, d = heapq.heappop(heap)
        if d < K:
            for lp, t in zip(logp[d], ids[d]):
                heapq.heappush(heap, (s - lp, t, len(scores), d + 1))
        scores.append(-s)
    return scores


def _philox_word(V, step, seq, key):
    """Word seq % 4 of Philox-4x32-10 (Salmon et al., SC 2011) for counters (v, step, seq // 4, 0), v < V."""
    mask = 0xFFFFFFFF

    def mulhilo(m, x):
        lo = (x & 0xFFFF) * m
        hi = (x >> 16) * m + (lo >> 16)
        return hi >> 16, ((hi & 0xFFFF) << 16) | (lo & 0xFFFF)

    z = torch.zeros(V, dtype=torch.int64, device="cuda")
    x = [torch.arange(V, dtype=torch.int64, device="cuda"), z + step, z + seq // 4, z]
    k0, k1 = key & mask, (key >> 32) & mask
    for _ in range(10):
        h0, l0 = mulhilo(0xD2511F53, x[0])
        h1, l1 = mulhilo(0xCD9E8D57, x[2])
        x = [h1 ^ x[1] ^ k0, l1, h0 ^ x[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return x[seq % 4]


def _exact_step(c, seed):
    w = _weights(c, seed)
    B, K, k, N = c["B"], c["K"], c["k"], c["N"]
    hid, u = _hidden(c, seed).double(), None
    if c["head"]:
        ids, h, S = _ids((B, K), c["V"], seed), torch.zeros(B, DS, dtype=torch.float64, device="cuda"), []
        for j in range(K):
            h = _gru_step(w, h, ids[:, j])
            S.append(h)
        u = _code(w, hid, torch.stack(S, 1)).view(B * K, R)
    lp = []
    for a in range(0, B * K, 256):
        b = min(B * K, a + 256)
        z = _logits(w, hid.view(B * K, -1)[a:b], None if u is None else u[a:b])
        v, i = z.topk(k, -1)
        lp.append((i, v - z.logsumexp(-1, keepdim=True)))
    ids, logp = (torch.cat(x).view(B, K, k) for x in zip(*lp))
    ci, cl = ids.cpu().tolist(), logp.cpu().tolist()
    score = torch.tensor([_tree_scores(ci[b], cl[b], N) for b in range(B)], dtype=torch.float64)
    return dict(topk_ids=None, topk_logp=logp, tree_parent=None, tree_token=None, tree_depth=None, tree_score=score)


def _exact_rollout(c, seed):
    w = _weights(c, seed)
    B, K, V = c["B"], c["K"], c["V"]
    hid = _hidden(c, seed).double()
    base = _logits({n: w[n] for n in ("w_lm",)}, hid.view(B * K, -1), None).view(B, K, V)
    uni = torch.rand(B, K, generator=_gen(seed, 34), device="cuda").double()
    h, t = torch.zeros(B, DS, dtype=torch.float64, device="cuda"), _ids((B,), V, seed)
    w2 = w["w2"].double()
    logp = torch.empty(B, K, dtype=torch.float64, device="cuda")
    for j in range(K):
        h = _gru_step(w, h, t)
        z = base[:, j] + _code(w, hid[:, j], h) @ w2.T + _bias(w, "b2")
        if c["rule"] == "cdf":
            cum = torch.softmax(z, -1).cumsum(-1)
            t = torch.searchsorted(cum, uni[:, j:j + 1] * cum[:, -1:], right=True).clamp_(max=V - 1).squeeze(-1)
        elif c["rule"] == "race":
            bits = torch.stack([_philox_word(V, j, b, int(seed) * 7919 + 1) for b in range(B)])
            t = (z - torch.log(-torch.log(((bits >> 9).double() + 0.5) / 2.0**23))).argmax(-1)
        else:
            t = z.argmax(-1)
        logp[:, j] = torch.log_softmax(z, -1).gather(1, t[:, None])[:, 0]
    return dict(tokens=None, logp=logp)


def exact(case, seed):
    if case["kind"] == "step":
        return _exact_step(case, seed)
    if case["kind"] == "rollout":
        return _exact_rollout(case, seed)
    return None  # verification returns whole numbers only
