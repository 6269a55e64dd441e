"""GPU parity of the fp32 head's kernels: the tiled CUDA-core linear layer (64 x 64 tiles, Kd
in steps of 32 split over four groups) at ragged and unaligned sizes, and whole fp32 networks at
the edges of the attention core (one node, narrow and 128-wide heads, head widths that leave
lanes idle, 512 nodes with few warps a CTA), against 64-bit references."""
import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_fused import _ll, _topk
from _helpers import TOL_VEC, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,Kd", [(1, 1, 1), (64, 64, 32), (65, 63, 31), (130, 72, 33),
                                    (1100, 200, 96), (2048, 256, 256), (70, 130, 68)])
@pytest.mark.parametrize("dt", [torch.float32, torch.bfloat16])
def test_linear_tiled(M, N, Kd, dt):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(M * 5 + N + Kd)
    A = torch.randn((M, Kd), generator=g, device="cuda").to(dt)
    W = torch.randn((N, Kd), generator=g, device="cuda").to(dt)
    bias = torch.randn(N, generator=g, device="cuda")
    res = torch.randn((M, N), generator=g, device="cuda")
    C = ll.test_linear(A, W, torch.float32, bias=bias, residual=res, path=1)
    want = A.double() @ W.double().T + bias + res
    # an fp32 sum of Kd + 2 terms: (Kd + 2) 2^-24 of the sum of their magnitudes
    tol = (Kd + 2) * 2.0 ** -24 * (A.double().abs() @ W.double().abs().T + 8).max().item()
    assert (C.double() - want).abs().max().item() <= tol


# clusters of 2, 4 and 8, uneven parts of Kd and a short last step, ragged tiles; path 0 where
# the rule takes another kernel (one wave of the split-N kernel, Kd below 256, more tiles than SMs)
@pytest.mark.parametrize("path,M,N,Kd", [(7, 1, 1, 64), (7, 65, 63, 36), (7, 64, 64, 2052),
                                         (7, 130, 260, 292), (7, 512, 512, 320), (7, 640, 256, 256),
                                         (0, 32, 256, 1024), (0, 64, 256, 4096), (0, 33, 256, 256),
                                         (0, 33, 256, 248), (0, 1000, 512, 264), (0, 1100, 96, 1000)])
@pytest.mark.parametrize("wdt", [torch.float32, torch.bfloat16])
def test_linear_tiled_split(path, M, N, Kd, wdt):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(M * 7 + N + Kd)
    A = torch.randn((M, Kd), generator=g, device="cuda")
    W = torch.randn((N, Kd), generator=g, device="cuda").to(wdt)
    bias = torch.randn(N, generator=g, device="cuda")
    res = torch.randn((M, N), generator=g, device="cuda")
    C = ll.test_linear(A, W, torch.float32, bias=bias, residual=res, path=path)
    want = A.double() @ W.double().T + bias + res
    # an fp32 sum of Kd + 2 terms, in any order
    tol = (Kd + 2) * 2.0 ** -24 * (A.double().abs() @ W.double().abs().T + 8).max().item()
    assert (C.double() - want).abs().max().item() <= tol


@pytest.mark.parametrize("B,L,K,D", [(1, 1, 1, 32), (2, 5, 7, 64), (9, 16, 8, 256), (1, 32, 16, 320),
                                     (2, 3, 3, 1024), (3, 17, 5, 96)])
def test_fp32_network_matches_oracle(B, L, K, D):
    _network_matches_oracle(B, L, K, D)


# the attention core's one query a warp (at most a wave of CTAs) and the sizes next to its edge:
# a last warp without a query, keys that fill no lane group, 8 heads x 19 CTAs of 152
@pytest.mark.parametrize("B,L,K,D", [(1, 1, 9, 64), (1, 11, 3, 96), (1, 19, 8, 256),
                                     (1, 17, 9, 256), (2, 9, 8, 64), (3, 7, 7, 32)])
def test_fp32_attention_one_query(B, L, K, D):
    _network_matches_oracle(B, L, K, D)


# more (sequence, head) pairs than SMs: a CTA of one warp, of two, of an odd number, of all eight
@pytest.mark.parametrize("B,L,K,D", [(20, 1, 3, 64), (24, 4, 2, 64), (20, 3, 3, 256), (21, 7, 3, 64),
                                     (20, 8, 4, 64)])
def test_fp32_attention_many_short_sequences(B, L, K, D):
    _network_matches_oracle(B, L, K, D)


def _network_matches_oracle(B, L, K, D):
    ll = _ll()
    wl = workloads.Workload(f"fp32_b{B}_l{L}_k{K}_d{D}", B=B, L=L, V=2000, K=K, d=D, H=128,
                            dtype="f32", logit_kind="normal_planted", logit_param=(3.0, 8.0),
                            seed_base=9950 + L * K)
    W = workloads.head_weights(wl)
    inp = workloads.batch_inputs(wl, wl.seeds())
    ids, logp = _topk(wl, inp["logits"])
    head = ll.Head.from_workload(wl, W, workloads.embed_table(wl.V, wl.H, wl.dtype))
    try:
        res = ll.embed_in_out(head, to_dev(ids.astype(np.int32), "f32"),
                              to_dev(logp.astype(np.float32), "f32"),
                              to_dev(inp["hidden"], wl.dtype), to_dev(inp["target"], wl.dtype))
        out, inn, anc = (t.cpu().numpy() for t in res)
    finally:
        head.close()
    for b in range(B):
        E = workloads.embed_rows(wl.V, wl.H, wl.dtype, ids[b].reshape(-1)).reshape(L, K, wl.H)
        o, i, a = oracle.head_forward(ids[b], logp[b].astype(np.float32).astype(np.float64),
                                      inp["hidden"][b], inp["target"][b], E, W)
        for got, want in ((out[b], o), (inn[b], i), (anc[b], a)):
            assert np.abs(got - want).max() <= TOL_VEC["f32"]
