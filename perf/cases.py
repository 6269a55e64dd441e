"""The work that a user of this library has it do, as cases that can be timed and compared.

Five families, each through the public calls of ``paper_2608_20530_gb300``:

``select``  the fused per-block selection (raw logits and hidden states to the scores the walk
            reads and the candidates), bf16 or fp32 heads;
``net``     the scoring network alone, for a program that has its candidates already
            (``embed_in_out``);
``topk``    the top-K + normaliser pass over logit rows (``topk_lse``);
``lm_head`` the LM-head projection fused with it (``lm_head_topk``);
``scores``  pair scores, the exact best path and the diagnostics along it, from vectors.

Shapes are the ones of this repository's workloads and of the paper's head (D = d = 1024,
L = 15, K = 8, H = 4096 or 2560), with ragged ones beside them. Weights are drawn once per
shape from a fixed seed, as a server loads one head; the seed of a case draws its inputs.
Token embeddings are at the hidden states' scale, so that candidates separate as they do under
a trained head. With ``graph`` the pass is captured once and replayed, as a serving loop does
for a batch size that it meets again and again; without it every pass is a plain call.
"""
import functools
import math

import numpy as np
import torch

import paper_2608_20530_gb300 as ll

V_FULL = 151936
N_HEADS, N_LAYERS, N_TGT = 8, 2, 5
SIGMA = 8.0


def _net(kind, name, B, D, L, K, H, V, dtype="bf16", logits="scaled", graph=False):
    return {"name": name, "kind": kind, "B": B, "D": D, "L": L, "K": K, "H": H, "V": V,
            "dtype": dtype, "logits": logits, "graph": graph}


def listed():
    return [
        # one request: a block of 16 slots, latency bound, replayed from a graph
        _net("select", "select_b1", 1, 256, 16, 8, 4096, V_FULL, logits="planted", graph=True),
        # 32 concurrent requests of mixed entropy
        _net("select", "select_b32", 32, 256, 16, 8, 4096, V_FULL, graph=True),
        # 64 requests with twice the candidates per slot
        _net("select", "select_k16_b64", 64, 256, 16, 16, 4096, V_FULL, logits="gumbel"),
        # the paper's own head for one request: 15 slots, width 1024
        _net("net", "net_d1024_b1", 1, 1024, 15, 8, 4096, V_FULL, graph=True),
        # the paper's smaller hidden width, two dozen requests
        _net("net", "net_d1024_b24", 24, 1024, 15, 8, 2560, 100003, graph=True),
        # 256 requests on a 512-wide head, 65,536 nodes
        _net("net", "net_d512_b256", 256, 512, 16, 16, 4096, V_FULL),
        # an fp32 head: a program that checks or trains against full precision
        _net("select", "select_f32_b16", 16, 256, 16, 8, 1024, 32000, dtype="f32", graph=True),
        # fp32 logits of an odd vocabulary (rows off 16-byte boundaries)
        {"name": "topk_f32_odd", "kind": "topk", "rows": 480, "V": 128257, "K": 10,
         "dtype": "f32", "logits": "scaled"},
        # 256 requests' logits on a coarse grid: many equal values around the K-th
        {"name": "topk_ties_4096", "kind": "topk", "rows": 4096, "V": V_FULL, "K": 16,
         "dtype": "bf16", "logits": "ties"},
        # the LM head of four requests' blocks: the weights' bytes bound it
        {"name": "lm_head_64", "kind": "lm_head", "rows": 64, "H": 4096, "V": V_FULL, "K": 8},
        # of about thirty: a ragged row count, the products bound it
        {"name": "lm_head_500", "kind": "lm_head", "rows": 500, "H": 4096, "V": V_FULL, "K": 8},
        # vectors to scores, best path, probabilities and acceptance of 200 requests
        {"name": "scores_b200", "kind": "scores", "B": 200, "L": 15, "K": 8, "d": 1024,
         "graph": True},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["select", "net", "topk", "lm_head", "scores"])
    if kind in ("select", "net"):
        f32 = rng.random() < 0.2
        D = rng.choice([64, 256]) if f32 else rng.choice([256, 256, 512, 1024])
        L = rng.randint(4, 16)
        K = rng.randint(2, 16)
        # at most the work of the largest listed case (its 65,536 nodes at D = 512)
        most = min(256, int((2048 if f32 else 32768) * (512 / D) ** 2 / (L * K)))
        return {"kind": kind, "B": _log_int(rng, 1, max(1, most)), "D": D, "L": L, "K": K,
                "H": rng.choice([1024, 2560, 4096]), "V": _log_int(rng, 8000, V_FULL),
                "dtype": "f32" if f32 else "bf16",
                "logits": rng.choice(["planted", "scaled", "gumbel", "ties"]),
                "graph": rng.random() < 0.5}
    if kind == "topk":
        f32 = rng.random() < 0.4
        return {"kind": kind, "rows": _log_int(rng, 1, 2000 if f32 else 4000),
                "V": _log_int(rng, 4000, V_FULL), "K": rng.randint(1, 32),
                "dtype": "f32" if f32 else "bf16",
                "logits": rng.choice(["planted", "scaled", "gumbel", "ties"])}
    if kind == "lm_head":
        return {"kind": kind, "rows": _log_int(rng, 1, 500), "H": 64 * rng.randint(8, 64),
                "V": _log_int(rng, 8000, V_FULL), "K": rng.randint(1, 16)}
    L, K = rng.randint(4, 16), rng.randint(2, 16)
    d = 4 * _log_int(rng, 16, 256)
    return {"kind": kind, "B": _log_int(rng, 1, max(2, min(256, 24_000_000 // (L * K * d)))),
            "L": L, "K": K, "d": d, "graph": rng.random() < 0.5}


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _tdt(case):
    return torch.float32 if case.get("dtype") == "f32" else torch.bfloat16


def _logits(case, lead, V, g):
    """Rows of logits: ``planted`` N(0, 3) with one +8 per row, ``scaled`` U[1, 5] * N(0, 1) per
    sequence, ``gumbel`` Gumbel / tau with tau 0.3, 1 or 3, ``ties`` 0.25 * round(N(0, 2) / 0.25)."""
    out = torch.empty((*lead, V), dtype=_tdt(case), device="cuda")
    rows = out.view(-1, V)
    for r0 in range(0, rows.shape[0], 256):
        n = min(256, rows.shape[0] - r0)
        x = torch.empty((n, V), device="cuda")
        kind = case["logits"]
        if kind == "gumbel":
            x.exponential_(generator=g).clamp_(min=1e-30).log_().neg_()
            taus = torch.tensor([0.3, 1.0, 3.0], device="cuda")
            x /= taus[torch.randint(0, 3, (n, 1), generator=g, device="cuda")]
        else:
            x.normal_(generator=g)
            if kind == "planted":
                x *= 3.0
                at = torch.randint(0, V, (n, 1), generator=g, device="cuda")
                x.scatter_add_(1, at, torch.full((n, 1), 8.0, device="cuda"))
            elif kind == "scaled":
                x *= 1.0 + 4.0 * torch.rand((n, 1), generator=g, device="cuda")
            else:
                x = torch.round(x * 8.0) * 0.25
        rows[r0:r0 + n] = x
    return out


def _weights(D, L, K, H, dtype):
    """The head's tensors on the device, in the storage type: N(0, 0.02), norm gains 1 + that."""
    g = _gen(1_000_003)
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    out = {}
    for name, shape in ll.blob_order(H, D, D, 2 * D, N_HEADS, L, K, N_LAYERS):
        a = 0.02 * torch.randn(shape, generator=g, device="cuda")
        if name in ("tgt_norm", "final_norm") or name.endswith((".an", ".fn")):
            a += 1.0
        out[name] = a.to(tdt)
    return out


def _table(V, H, dtype):
    """The frozen token-embedding table [V, H], N(0, 1)."""
    g = _gen(1_000_033)
    out = torch.empty((V, H), dtype=torch.float32 if dtype == "f32" else torch.bfloat16,
                      device="cuda")
    for r in range(0, V, 16384):
        n = min(16384, V - r)
        out[r:r + n] = torch.randn((n, H), generator=g, device="cuda")
    return out


@functools.lru_cache(maxsize=1)
def _head(D, L, K, H, V, dtype):
    """The head that a server loads once and keeps."""
    W = {k: v.float().cpu().numpy() for k, v in _weights(D, L, K, H, dtype).items()}
    E = _table(V, H, dtype).cpu()
    E = E.numpy() if dtype == "f32" else E.view(torch.int16).numpy().view(np.uint16)
    return ll.Head(H=H, D=D, d=D, n_heads=N_HEADS, ffn=2 * D, n_layers=N_LAYERS, L=L, K=K, V=V,
                   n_tgt=N_TGT, dtype=dtype, weights=W, embed_table=E)


def _inputs(case, seed):
    g, c, tdt = _gen(seed), case, _tdt(case)
    if c["kind"] in ("select", "net"):
        B, L, H = c["B"], c["L"], c["H"]
        x = {"hidden": torch.randn((B, L, H), generator=g, device="cuda").to(tdt),
             "target": torch.randn((B, N_TGT, H), generator=g, device="cuda").to(tdt)}
        if c["kind"] == "select":
            x["logits"] = _logits(c, (B, L), c["V"], g)
        else:                                     # candidates as a top-K pass leaves them
            x["ids"] = torch.randint(0, c["V"], (B, L, c["K"]), generator=g, device="cuda",
                                     dtype=torch.int32)
            gap = torch.empty((B, L, c["K"]), device="cuda").exponential_(generator=g)
            x["logp"] = -torch.cumsum(gap, -1)
        return x
    if c["kind"] == "topk":
        return {"logits": _logits(c, (c["rows"],), c["V"], g)}
    if c["kind"] == "lm_head":
        w = torch.empty((c["V"], c["H"]), dtype=tdt, device="cuda")
        for r in range(0, c["V"], 16384):
            n = min(16384, c["V"] - r)
            w[r:r + n] = 0.02 * torch.randn((n, c["H"]), generator=g, device="cuda")
        return {"hidden": torch.randn((c["rows"], c["H"]), generator=g, device="cuda").to(tdt),
                "w": w}
    B, L, K, d = c["B"], c["L"], c["K"], c["d"]
    # vectors with a part in common along the block, as neighbouring candidates have
    base = torch.randn((B, 1, 1, d), generator=g, device="cuda")
    ids = torch.randint(0, V_FULL, (B, L, K), generator=g, device="cuda", dtype=torch.int32)
    at = torch.randint(0, K, (B, L, 1), generator=g, device="cuda")
    return {"out": base + torch.randn((B, L, K, d), generator=g, device="cuda"),
            "in": base + torch.randn((B, L, K, d), generator=g, device="cuda"),
            "anchor": base[:, 0, 0] + torch.randn((B, d), generator=g, device="cuda"),
            "ids": ids, "truth": torch.gather(ids, 2, at)[..., 0].contiguous()}


def _call(s):
    c, x = s["case"], s["x"]
    if c["kind"] == "select":
        # the scores and candidates the block is chosen from; the tokens only where fp32 leaves
        # no doubt about them (a bf16 head's closest runners-up lie within its rounding)
        tokens = ll.select_block(s["head"], x["logits"], x["hidden"], x["target"], ws=s["ws"],
                                 tokens=s["tokens"])
        out = dict(s["views"])
        if c["dtype"] == "f32":
            out["tokens"] = tokens
        return out
    if c["kind"] == "net":
        out, inn, anc = ll.embed_in_out(s["head"], x["ids"], x["logp"], x["hidden"], x["target"],
                                        ws=s["ws"])
        return {"out": out, "in": inn, "anchor": anc}
    if c["kind"] == "topk":
        ids, logp, lse = ll.topk_lse(x["logits"], c["K"], ws=s["ws"])
        return {"ids": ids, "logp": logp, "lse": lse}
    if c["kind"] == "lm_head":
        ids, logp, lse = ll.lm_head_topk(x["hidden"], x["w"], c["K"], ws=s["ws"])
        return {"ids": ids, "logp": logp, "lse": lse}
    A, P = ll.pair_scores(x["out"], x["in"], x["anchor"])
    choice, tokens, score = ll.best_path(A, P, x["ids"], SIGMA)
    pa, pp = ll.local_softmax(A, P, SIGMA)
    prob, gap, lp = ll.path_probs(A, P, choice, SIGMA)
    covered, prefix, acc = ll.block_acceptance(x["ids"], tokens, x["truth"])
    return {"A": A, "P": P, "choice": choice, "tokens": tokens, "score": score, "pa": pa,
            "pp": pp, "prob": prob, "gap": gap, "lp": lp, "covered": covered, "prefix": prefix,
            "acc": acc}


def prepare(case, seed):
    c = dict(case)
    s = {"case": c, "x": _inputs(c, seed)}
    if c["kind"] in ("select", "net"):
        s["head"] = _head(c["D"], c["L"], c["K"], c["H"], c["V"], c["dtype"])
        s["ws"] = s["head"].workspace(c["B"])
        if c["kind"] == "select":
            s["tokens"] = torch.empty((c["B"], c["L"]), dtype=torch.int32, device="cuda")
            views = ll.select_block_intermediates(s["head"], c["B"], s["ws"])
            s["views"] = {k: views[k] for k in ("ids", "logp", "lse", "A", "P")}
    elif c["kind"] == "topk":
        n = int(ll.lib().lilicorr_topk_lse_workspace_bytes(c["rows"], c["V"], c["K"]))
        s["ws"] = ll.Workspace(n)
    elif c["kind"] == "lm_head":
        n = int(ll.lib().lilicorr_lm_head_topk_workspace_bytes(c["rows"], c["H"], c["V"], c["K"]))
        s["ws"] = ll.Workspace(n)
    if c.get("graph"):
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _call(s)                              # first-use setup stays out of the capture
        torch.cuda.current_stream().wait_stream(side)
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            s["outputs"] = _call(s)
    return s


def run(state):
    if "graph" in state:
        state["graph"].replay()
        return state["outputs"]
    return _call(state)


# ------------------------------------------------------------------------------ work, limits
def work(case):
    c = case
    if c["kind"] == "topk":
        es = 4 if c["dtype"] == "f32" else 2
        return {"bytes": c["rows"] * (c["V"] * es + c["K"] * 8 + 4), "flops": 3 * c["rows"] * c["V"]}
    if c["kind"] == "lm_head":
        return {"bytes": 2 * c["H"] * (c["V"] + c["rows"]) + c["rows"] * (c["K"] * 8 + 4),
                "flops": 2 * c["rows"] * c["H"] * c["V"]}
    B, L, K = c["B"], c["L"], c["K"]
    pairs = B * ((L - 1) * K * K + K)
    if c["kind"] == "scores":
        n, d = B * L * K, c["d"]
        # vectors and ids in; A and P once more as probabilities; paths, gaps and coverage
        return {"bytes": 4 * d * (2 * n + B) + 4 * n + 8 * pairs + 4 * B * (7 * L + 4),
                "flops": 2 * d * pairs + 4 * d * n + 8 * pairs}
    es, D, H, n = (4 if c["dtype"] == "f32" else 2), c["D"], c["H"], B * L * K
    weights = es * D * (2 * H + 8 * N_LAYERS * D + 7 * D)
    flops = 2 * D * H * B * (L + 1) + n * D * (2 * D + 16 * N_LAYERS * D + 4 * D + 4 * D + 10)
    flops += 4 * D * B * D + 4 * N_LAYERS * n * L * K * D
    by = weights + es * H * B * (L + N_TGT) + 4 * n * D
    if c["kind"] == "net":
        return {"bytes": by + 8 * n + 4 * D * (2 * n + B), "flops": flops}
    by += es * B * L * c["V"] + 8 * n + 4 * B * L + 4 * pairs
    return {"bytes": by, "flops": flops + 2 * D * pairs}


def tolerance(case):
    # About four times the error against exact() that was measured on a GB300.
    if case["kind"] == "topk":                    # one fp32 normaliser per row: 1.3e-7
        return {"rel": 6e-7}
    if case["kind"] == "lm_head":                 # fp32 sums of up to 4096 products: 2.2e-6;
        return {"rel": 9e-6, "differ": 2e-3}      # the closest logits may change places
    if case["kind"] == "scores":                  # differences of cosines (gap): 3.4e-6
        return {"rel": 1.4e-5, "differ": 5e-3}
    if case["dtype"] == "f32":                    # some ten fp32 products in a row: 1e-6
        return {"rel": 5e-6, "differ": 5e-3}
    return {"rel": 0.016, "max": 0.2}             # the same with bf16 operands: 4e-3


# ------------------------------------------------------------------------------ 64 bits
def _exact_topk(rows, K):
    """Top-K (larger first, then lower id), log-probs and normaliser of float64 rows."""
    top, logp, lse = [], [], []
    for r in rows.split(256):
        x = r.double()
        v, i = torch.sort(x, dim=-1, descending=True, stable=True)
        z = torch.logsumexp(x, -1)
        top.append(i[:, :K])
        logp.append(v[:, :K] - z[:, None])
        lse.append(z)
    return torch.cat(top), torch.cat(logp), torch.cat(lse)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True).clamp_min(1e-12)


def _rms(x, gain):
    return x * torch.rsqrt((x * x).mean(-1, keepdim=True) + 1e-6) * gain


def _silu(x):
    return x * torch.sigmoid(x)


def _exact_net(c, x, ids, logp):
    """Unit out and in vectors [B, L, K, D] and anchors [B, D] in float64."""
    W = {k: v.double() for k, v in _weights(c["D"], c["L"], c["K"], c["H"], c["dtype"]).items()}
    B, L, K, D = c["B"], c["L"], c["K"], c["D"]
    lin = lambda a, n: a @ W[n + "_w"].T + W[n + "_b"]  # noqa: E731
    E = _table(c["V"], c["H"], c["dtype"])
    emb = torch.cat([lin(E[i].double(), "emb") for i in ids.reshape(-1).long().split(8192)])
    hid = lin(x["hidden"].double(), "hid")
    k = torch.arange(K, device="cuda", dtype=torch.float64)
    # the five confidence scalars: log-probability, probability, gap to the slot's first
    # candidate, rank scaled to [0, 1], whether it is the first
    f = torch.stack([logp, logp.exp(), logp[..., :1] - logp, (k / max(K - 1, 1)).expand_as(logp),
                     (k == 0).double().expand_as(logp)], -1)
    conf = _silu(f @ W["conf1_w"].T + W["conf1_b"]) @ W["conf2_w"].T + W["conf2_b"]
    h = emb.view(B, L, K, D) + hid[:, :, None] + conf + W["slot"][:, None] + W["rank"]
    h = h.reshape(B, L * K, D)
    t = _rms(x["target"].double().mean(1), W["tgt_norm"]) @ W["tgt_w"].T + W["tgt_b"]
    slot = torch.arange(L * K, device="cuda") // K
    rel = slot[None, :] - slot[:, None]
    hd = D // N_HEADS
    for i in range(N_LAYERS):
        w = lambda n: W["l%d.%s" % (i, n)]  # noqa: E731
        a = _rms(h, w("an"))
        q, k, v = ((a @ w("w" + n).T + w("b" + n)).view(B, L * K, N_HEADS, hd).transpose(1, 2)
                   for n in "qkv")
        bias = w("dist")[:, rel + L - 1] + w("same")[:, None, None] * (rel == 0)
        att = torch.cat([torch.softmax(qq @ kk.transpose(-1, -2) / math.sqrt(hd) + bias, -1) @ vv
                         for qq, kk, vv in zip(q.split(16), k.split(16), v.split(16))])
        h = h + att.transpose(1, 2).reshape(B, L * K, D) @ w("wo").T + w("bo")
        h = h + _silu(_rms(h, w("fn")) @ w("w1").T + w("b1")) @ w("w2").T + w("b2")
    h = _rms(h, W["final_norm"])
    tt = t[:, None].expand_as(h)
    u = _silu(torch.cat([h, tt, h * tt], -1) @ W["fuse_w"].T + W["fuse_b"])
    shape = (B, L, K, D)
    return _unit(lin(u, "out")).view(shape), _unit(lin(u, "in")).view(shape), _unit(lin(t, "anc"))


def _exact_pairs(out, inn, anchor):
    out, inn, anchor = _unit(out), _unit(inn), _unit(anchor)
    return (torch.einsum("bd,bkd->bk", anchor, inn[:, 0]),
            torch.einsum("bskd,bsjd->bskj", out[:, :-1], inn[:, 1:]))


def exact(case, seed):
    c, x = dict(case), _inputs(case, seed)
    if c["kind"] == "topk":
        _, logp, lse = _exact_topk(x["logits"], c["K"])
        return {"ids": None, "logp": logp, "lse": lse}
    if c["kind"] == "lm_head":
        h = x["hidden"].double()
        z = torch.cat([h @ w.double().T for w in x["w"].split(16384)], 1)
        v, lse = torch.topk(z, c["K"], dim=-1)[0], torch.logsumexp(z, -1)
        return {"ids": None, "logp": v - lse[:, None], "lse": lse}
    if c["kind"] == "net":
        out, inn, anc = _exact_net(c, x, x["ids"], x["logp"].double())
        return {"out": out, "in": inn, "anchor": anc}
    if c["kind"] == "select":
        B, L, K = c["B"], c["L"], c["K"]
        ids, logp, lse = _exact_topk(x["logits"].view(B * L, -1), K)
        logp = logp.view(B, L, K)
        A, P = _exact_pairs(*_exact_net(c, x, ids.view(B, L, K), logp))
        out = {"ids": None, "logp": logp, "lse": lse.view(B, L), "A": A, "P": P}
        if c["dtype"] == "f32":
            out["tokens"] = None
        return out
    A, P = _exact_pairs(x["out"].double(), x["in"].double(), x["anchor"].double())
    # the best path, left to right, and the values along it
    B, K = A.shape
    score, back = SIGMA * A, []
    for s in range(P.shape[1]):
        best, frm = (score[:, :, None] + SIGMA * P[:, s]).max(1)
        score = best
        back.append(frm)
    total, at = score.max(-1)
    path = [at]
    for frm in reversed(back):
        at = torch.gather(frm, 1, at[:, None])[:, 0]
        path.append(at)
    path = torch.stack(path[::-1], 1)
    pa, pp = torch.softmax(SIGMA * A, -1), torch.softmax(SIGMA * P, -1)
    b = torch.arange(B, device="cuda")
    prob, gap = [], []
    for s in range(path.shape[1]):
        z = SIGMA * (A if s == 0 else P[b, s - 1, path[:, s - 1]])
        q = torch.softmax(z, -1)
        prob.append(q[b, path[:, s]])
        rest = z.clone()
        rest[b, path[:, s]] = -math.inf
        gap.append(z[b, path[:, s]] - rest.max(-1)[0])
    prob, gap = torch.stack(prob, 1), torch.stack(gap, 1)
    return {"A": A, "P": P, "choice": None, "tokens": None, "score": total, "pa": pa, "pp": pp,
            "prob": prob, "gap": gap, "lp": prob.log().sum(1), "covered": None, "prefix": None,
            "acc": None}
