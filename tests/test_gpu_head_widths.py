"""Heads of unusual widths against the oracle. Vectors narrower or wider than the network (d != D): the
anchor product (N = d) and the fusion layer's t product (N = D) share a launch whose grid is the
wider one's, on the few-row kernel (1, 4 and 16 requests) and on the row-block kernel (more). The
widest networks build their nodes in parts, whatever the number of slots."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_fused import _ll
from _helpers import TOL_VEC, to_dev

pytestmark = pytest.mark.gpu


# widths that end inside a block of 4 or 32 columns' grid; fp32 heads take the row-block kernel below 256
@pytest.mark.parametrize("B,D,d,dtype", [
    (1, 128, 40, "bf16"), (4, 128, 200, "bf16"), (16, 64, 136, "f32"), (17, 128, 40, "bf16"),
    (33, 128, 200, "bf16"), (20, 64, 24, "f32"), (18, 64, 104, "f32"), (3, 256, 96, "bf16"),
    (40, 256, 320, "bf16"), (19, 256, 72, "f32"), (1, 256, 264, "f32")])
def test_vectors_of_another_width(B, D, d, dtype):
    _network_matches_oracle(B, 3, 4, D, d, 2 * D, 8, 2, dtype, 0.05)


# more slots than two CTAs an SM, the widths next to what one CTA stages, and twice that
@pytest.mark.parametrize("B,L,D,dtype", [(20, 16, 1984, "f32"), (20, 16, 2048, "bf16"),
                                         (1, 2, 2048, "f32"), (20, 16, 4096, "f32")])
def test_wide_networks(B, L, D, dtype):
    _network_matches_oracle(B, L, 2, D, 64, 64, D // 64, 1, dtype, 0.02)


def _network_matches_oracle(B, L, K, D, d, F, heads, layers, dtype, std):
    ll = _ll()
    V, H, tgt = 300, 64, 5
    rng = np.random.default_rng(D * 7 + d + B)

    def stored(a):                                # the value a head of this type holds
        t = torch.from_numpy(np.ascontiguousarray(a, np.float32))
        return (t.to(torch.bfloat16).float() if dtype == "bf16" else t).numpy()

    W = {}
    for name, shape in ll.blob_order(H, D, d, F, heads, L, K, layers):
        gain = name in ("tgt_norm", "final_norm") or name.endswith((".an", ".fn"))
        W[name] = stored(std * rng.standard_normal(shape) + (1.0 if gain else 0.0))
    E, hidden, target = (stored(rng.standard_normal(s)) for s in ((V, H), (B, L, H), (B, tgt, H)))
    ids = np.stack([[rng.permutation(V)[:K] for _ in range(L)] for _ in range(B)])
    logp = -np.cumsum(rng.exponential(size=(B, L, K)), -1).astype(np.float32)
    Eh = (E.view(np.uint32) >> 16).astype(np.uint16) if dtype == "bf16" else E
    head = ll.Head(H=H, D=D, d=d, n_heads=heads, ffn=F, n_layers=layers, L=L, K=K, V=V, n_tgt=tgt,
                   dtype=dtype, weights=W, embed_table=Eh)
    try:
        ws = head.workspace(B)
        res = [t.cpu().numpy() for t in ll.embed_in_out(
            head, to_dev(ids.astype(np.int32), "f32"), to_dev(logp, "f32"), to_dev(hidden, dtype),
            to_dev(target, dtype), ws=ws)]
        assert ws.status() == 0
    finally:
        head.close()
    for b in {0, B // 2, B - 1}:
        want = oracle.head_forward(ids[b], logp[b].astype(np.float64), hidden[b], target[b],
                                   E[ids[b].reshape(-1)].reshape(L, K, H), W, n_heads=heads,
                                   n_layers=layers)
        for got, w in zip((res[0][b], res[1][b], res[2][b]), want):
            assert got.shape == w.shape
            assert np.abs(got - w).max() <= TOL_VEC[dtype]
