"""Which kernel the network's rule gives a bf16 product of more than 64 rows, seen by its sums (the
kernels add Kd up in different orders): short Kd and many tiles stay with the whole-K and the
persistent kernel, where Kd split over a cluster is slower; and heads of small width, whose
products are all of that kind, against the oracle."""
import numpy as np
import pytest
import torch

import workloads
from test_gpu_fused import _ll, _oracle_check, _topk
from _helpers import to_dev

pytestmark = pytest.mark.gpu

SMALL, TC, SPLIT = 4, 3, 6


@pytest.mark.parametrize("M,N,Kd,dt,path", [
    (65, 256, 256, torch.float32, SMALL), (128, 1536, 256, torch.bfloat16, SMALL),
    (128, 512, 512, torch.bfloat16, SMALL), (120, 3072, 512, torch.float32, SMALL),
    (120, 512, 512, torch.float32, SPLIT), (129, 512, 256, torch.float32, TC),
    (2048, 256, 256, torch.bfloat16, TC), (360, 512, 512, torch.bfloat16, SPLIT),
    (480, 1024, 512, torch.float32, SPLIT), (480, 1024, 512, torch.bfloat16, TC),
    (1024, 1024, 512, torch.float32, TC), (1024, 1024, 1024, torch.bfloat16, TC),
    (1024, 1024, 1024, torch.float32, SPLIT), (720, 1024, 2048, torch.bfloat16, SPLIT)])
def test_rule(M, N, Kd, dt, path):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(M + N + Kd)
    A = torch.randn((M, Kd), generator=g, device="cuda").to(torch.bfloat16)
    W = (0.02 * torch.randn((N, Kd), generator=g, device="cuda")).to(torch.bfloat16)
    assert torch.equal(ll.test_linear(A, W, dt, path=0), ll.test_linear(A, W, dt, path=path))


# widths whose heads are narrower than the tensor cores' attention takes, and one with five chunks
@pytest.mark.parametrize("B,L,K,D", [(1, 8, 8, 64), (2, 15, 8, 64), (16, 4, 2, 128), (2, 8, 8, 128),
                                     (3, 16, 16, 128), (1, 15, 8, 320), (5, 8, 8, 320)])
def test_narrow_network_matches_oracle(B, L, K, D):
    ll = _ll()
    wl = workloads.Workload(f"narrow_b{B}_l{L}_k{K}_d{D}", B=B, L=L, V=2000, K=K, d=D, H=256,
                            dtype="bf16", logit_kind="normal_planted", logit_param=(3.0, 8.0),
                            seed_base=9700 + L * K)
    W = workloads.head_weights(wl)
    inp = workloads.batch_inputs(wl, wl.seeds())
    ids, logp = _topk(wl, inp["logits"])
    head = ll.Head.from_workload(wl, W, workloads.embed_table(wl.V, wl.H, wl.dtype))
    try:
        ws = head.workspace(B)
        res = [t.cpu().numpy() for t in ll.embed_in_out(
            head, to_dev(ids.astype(np.int32), "f32"), to_dev(logp.astype(np.float32), "f32"),
            to_dev(inp["hidden"], wl.dtype), to_dev(inp["target"], wl.dtype), ws=ws)]
        assert ws.status() == 0
        _oracle_check(wl, W, inp, ids, logp, *res, range(B))
    finally:
        head.close()


# up to 64 nodes: few-row products, folded from five nodes on where Kd splits over four CTAs
@pytest.mark.parametrize("B,L,K,D", [(1, 64, 1, 256), (1, 4, 1, 512), (1, 2, 2, 1024), (1, 5, 1, 512),
                                     (3, 4, 4, 384), (2, 5, 3, 320), (1, 64, 1, 320)])
def test_network_of_few_nodes_matches_oracle(B, L, K, D):
    test_narrow_network_matches_oracle(B, L, K, D)
