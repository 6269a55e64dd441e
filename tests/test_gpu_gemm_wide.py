"""GPU parity of the tensor-core linear layer's 128-wide stages (bf16 outputs, 256-column tiles)
and its fp32 neighbours at the edges of their tiles: a ragged last row tile, ragged columns, Kd of
one chunk, an odd number of chunks, no whole chunks, against 64-bit products; and networks whose
products all run on it, with the RMSNorms folded into them, against the oracle."""
import numpy as np
import pytest
import torch

import workloads
from test_gpu_fused import _ll, _oracle_check, _topk
from _helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,Kd", [(20000, 256, 64), (19585, 256, 512), (19713, 264, 192),
                                    (9000, 600, 72), (5120, 1536, 1024), (40000, 512, 320)])
def test_linear_wide_stages(M, N, Kd):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(M + N + Kd)
    A = torch.randn((M, Kd), generator=g, device="cuda").to(torch.bfloat16)
    W = (0.05 * torch.randn((N, Kd), generator=g, device="cuda")).to(torch.bfloat16)
    bias = torch.randn(N, generator=g, device="cuda")
    res = torch.randn((M, N), generator=g, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    prod = A.double() @ W.double().T
    # fp32 sums of Kd bf16 products: Kd * 2^-23 of the sum of magnitudes bounds them
    tol = Kd * 2.0 ** -23 * (A[:512].double().abs() @ W.double().abs().T).max().item() * 2 + 1e-5
    for b, r, odt in [(None, None, torch.float32), (bias, res, torch.float32),
                      (bias, None, torch.bfloat16)]:
        C = ll.test_linear(A, W, odt, bias=b, residual=r, path=3, status=status)
        want = prod if b is None else prod + b
        want = want if r is None else want + r
        rnd = 2.0 ** -8 * want.abs() if odt == torch.bfloat16 else 0.0
        assert ((C.double() - want).abs() - rnd).max().item() <= tol, odt
    assert int(status.item()) == 0


# 256-column tiles; then 192-column ones, whose last is past N in part (1024 = 5 x 192 + 64, 512 =
# 2 x 192 + 128), with row tiles that span sequences: 2880 rows x 1024 and 12,000 x 512
@pytest.mark.parametrize("B,L,K,D", [(90, 15, 15, 512), (80, 16, 8, 1024), (24, 15, 8, 1024),
                                     (100, 15, 8, 512)])
def test_wide_network_matches_oracle(B, L, K, D):
    ll = _ll()
    wl = workloads.Workload(f"wide_b{B}_d{D}", B=B, L=L, V=1000, K=K, d=D, H=64, dtype="bf16",
                            logit_kind="normal_planted", logit_param=(3.0, 8.0), seed_base=9800)
    W = workloads.head_weights(wl)
    inp = workloads.batch_inputs(wl, wl.seeds())
    ids, logp = _topk(wl, inp["logits"])
    head = ll.Head.from_workload(wl, W, workloads.embed_table(wl.V, wl.H, wl.dtype))
    try:
        args = [to_dev(ids.astype(np.int32), "f32"), to_dev(logp.astype(np.float32), "f32"),
                to_dev(inp["hidden"], wl.dtype), to_dev(inp["target"], wl.dtype)]
        ws = head.workspace(B)
        res = [t.cpu().numpy() for t in ll.embed_in_out(head, *args, ws=ws)]
        again = [t.cpu().numpy() for t in ll.embed_in_out(head, *args, ws=ws)]
        assert ws.status() == 0
        for a, b in zip(res, again):
            assert np.array_equal(a, b)
        _oracle_check(wl, W, inp, ids, logp, *res, (0, 1, B // 2, B - 1))
    finally:
        head.close()
