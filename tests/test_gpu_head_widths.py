"""Heads whose vectors are narrower or wider than the network (d != D): the anchor product (N = d) and
the fusion layer's t product (N = D) share a launch whose grid is the wider one's, on the few-row
kernel (1, 4 and 16 requests) and on the row-block kernel (more), against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_fused import _ll
from _helpers import TOL_VEC, to_dev

pytestmark = pytest.mark.gpu


# widths that end inside a block of 4 or 32 columns' grid; fp32 heads take the row-block kernel below 256
@pytest.mark.parametrize("B,D,d,dtype", [
    (1, 128, 40, "bf16"), (4, 128, 200, "bf16"), (16, 64, 136, "f32"), (17, 128, 40, "bf16"),
    (33, 128, 200, "bf16"), (20, 64, 24, "f32"), (18, 64, 104, "f32"), (3, 256, 96, "bf16"),
    (40, 256, 320, "bf16"), (19, 256, 72, "f32"), (1, 256, 264, "f32")])
def test_vectors_of_another_width(B, D, d, dtype):
    ll = _ll()
    L, K, V, H, heads, tgt = 3, 4, 300, 64, 8, 5
    rng = np.random.default_rng(D * 7 + d + B)

    def stored(a):                                # the value a head of this type holds
        t = torch.from_numpy(np.ascontiguousarray(a, np.float32))
        return (t.to(torch.bfloat16).float() if dtype == "bf16" else t).numpy()

    W = {}
    for name, shape in ll.blob_order(H, D, d, 2 * D, heads, L, K, 2):
        gain = name in ("tgt_norm", "final_norm") or name.endswith((".an", ".fn"))
        W[name] = stored(0.05 * rng.standard_normal(shape) + (1.0 if gain else 0.0))
    E, hidden, target = (stored(rng.standard_normal(s)) for s in ((V, H), (B, L, H), (B, tgt, H)))
    ids = np.stack([[rng.permutation(V)[:K] for _ in range(L)] for _ in range(B)])
    logp = -np.cumsum(rng.exponential(size=(B, L, K)), -1).astype(np.float32)
    Eh = (E.view(np.uint32) >> 16).astype(np.uint16) if dtype == "bf16" else E
    head = ll.Head(H=H, D=D, d=d, n_heads=heads, ffn=2 * D, n_layers=2, L=L, K=K, V=V, n_tgt=tgt,
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
                                   E[ids[b].reshape(-1)].reshape(L, K, H), W)
        for got, w in zip((res[0][b], res[1][b], res[2][b]), want):
            assert got.shape == w.shape
            assert np.abs(got - w).max() <= TOL_VEC[dtype]
