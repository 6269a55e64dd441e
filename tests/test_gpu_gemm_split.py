"""GPU parity of the products with few output tiles (Kd split over a thread-block cluster,
partial sums added through distributed shared memory): one linear layer against fp32 PyTorch
at the edges of its tiles and splits, and whole scoring networks whose products, with the
RMSNorms folded into them, all run on it, against the fp64 oracle."""
import numpy as np
import pytest
import torch

import workloads
from test_gpu_fused import _ll, _oracle_check, _topk
from _helpers import to_dev

pytestmark = pytest.mark.gpu

CASES = [  # M, N, Kd: one and several row tiles, ragged columns, 1 to 8 ways, uneven parts
    (5, 8, 64), (15, 1024, 4096), (120, 3072, 1024), (128, 64, 8), (129, 72, 136), (37, 200, 1096),
    (512, 256, 4096), (24, 1024, 2560), (1, 64, 512), (300, 192, 1024),
]


@pytest.mark.parametrize("M,N,Kd", CASES)
def test_linear_split(M, N, Kd):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(M * 7 + N + Kd)
    A = torch.randn((M, Kd), generator=g, device="cuda").to(torch.bfloat16)
    W = (0.02 * torch.randn((N, Kd), generator=g, device="cuda")).to(torch.bfloat16)
    bias = 0.1 * torch.randn(N, generator=g, device="cuda")
    res = torch.randn((M, N), generator=g, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for act, b, r, odt in [(0, None, None, torch.float32), (1, bias, None, torch.float32),
                           (0, bias, res, torch.float32), (1, bias, None, torch.bfloat16)]:
        C = ll.test_linear(A, W, odt, bias=b, residual=r, act=act, path=6, status=status)
        again = ll.test_linear(A, W, odt, bias=b, residual=r, act=act, path=6, status=status)
        torch.cuda.synchronize()
        want = A.double() @ W.double().T
        # fp32 sums of Kd bf16 products: Kd * 2^-24 of the sum of magnitudes bounds them
        tol = Kd * 2.0 ** -23 * (A.double().abs() @ W.double().abs().T).max().item() + 1e-6
        want = want if b is None else want + b
        if act:
            # __expf (2 ulp) and, for bf16, tanh.approx (2^-11) and the rounding (2^-9)
            want = torch.nn.functional.silu(want)
            tol = tol * 1.1 + want.abs().max().item() * (2.0 ** -8 if odt == torch.bfloat16
                                                         else 2.0 ** -20)
        want = want if r is None else want + r
        assert (C.double() - want).abs().max().item() <= tol, (act, odt)
        assert torch.equal(C, again)
    assert int(status.item()) == 0


def test_linear_split_refuses_many_tiles():
    ll = _ll()
    A = torch.zeros((4096, 64), dtype=torch.bfloat16, device="cuda")
    W = torch.zeros((512, 64), dtype=torch.bfloat16, device="cuda")
    with pytest.raises(ll.LilicorrError):
        ll.test_linear(A, W, path=6)


# the paper's head for one request; few nodes; a width of five column tiles (their sums of
# squares are no multiple of four slots); several row tiles, some products on each kernel
@pytest.mark.parametrize("B,L,K,D", [(1, 15, 8, 1024), (1, 3, 3, 512), (2, 16, 8, 320),
                                     (5, 16, 16, 512), (3, 5, 7, 1024)])
def test_split_network_matches_oracle(B, L, K, D):
    ll = _ll()
    wl = workloads.Workload(f"split_b{B}_l{L}_k{K}_d{D}", B=B, L=L, V=2000, K=K, d=D, H=256,
                            dtype="bf16", logit_kind="normal_planted", logit_param=(3.0, 8.0),
                            seed_base=9900 + L * K)
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
        assert np.allclose(np.linalg.norm(res[0], axis=-1), 1, atol=1e-5)
        _oracle_check(wl, W, inp, ids, logp, *res, range(B))
    finally:
        head.close()
