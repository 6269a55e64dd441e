"""The failure side of the bounded waits in the kernels whose CTAs work in clusters, as
test_gpu_timeout.py has it for the persistent product: copies withheld in every CTA, or in one CTA of
each cluster while its peers go on, must end in the timeout status in the time that the limits give,
with the context usable and the next call right."""
import time

import pytest
import torch

from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu

TIMEOUT = 6        # LILICORR_ERR_TIMEOUT
LIMIT = 2_000_000  # about 1 ms of SM cycles per wait


# one CTA a tile, two, four and eight; few-row sums (at most 64 rows) and the others, with more chunks
# a CTA than stages and with fewer
@pytest.mark.parametrize("M,N,Kd", [(16, 128, 4096), (48, 1024, 1024), (20, 64, 64), (128, 64, 192),
                                    (200, 512, 512), (360, 1024, 2560), (300, 192, 1024)])
@pytest.mark.parametrize("first_only", [False, True])
def test_split_product_times_out(M, N, Kd, first_only):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(M + N)
    A = torch.randn((M, Kd), generator=g, device="cuda").to(torch.bfloat16)
    W = (0.05 * torch.randn((N, Kd), generator=g, device="cuda")).to(torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    want = A.double() @ W.double().T
    torch.cuda.synchronize()
    for _ in range(2):
        t0 = time.perf_counter()
        ll.test_linear_split_timeout(A, W, LIMIT, status, first_only)
        torch.cuda.synchronize()
        dt = time.perf_counter() - t0
        assert int(status.item()) == TIMEOUT
        assert dt < 5.0, f"the timed-out launch took {dt:.2f} s"
        status.zero_()
        C = ll.test_linear(A, W, path=6, status=status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        # fp32 sums of Kd bf16 products: Kd * 2^-23 of the sum of magnitudes bounds them
        tol = Kd * 2.0 ** -23 * (A.double().abs() @ W.double().abs().T).max().item() + 1e-6
        assert (C.double() - want).abs().max().item() <= tol


def test_split_hook_rejects_unbounded_limits():
    ll = _ll()
    A = torch.zeros((128, 64), device="cuda", dtype=torch.bfloat16)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    for bad in (0, 10, 10**12):
        with pytest.raises(ll.LilicorrError):
            ll.test_linear_split_timeout(A, A, bad, status)


# a tile a pair and several, whole steps of H and a last one of half, a pair whose second CTA has no rows
@pytest.mark.parametrize("rows,H,V,K", [(129, 2048, 257, 4), (256, 2112, 39000, 8),
                                        (257, 2048, 9000, 8), (400, 4096, 40000, 16)])
@pytest.mark.parametrize("second_only", [False, True])
def test_lm_head_pair_times_out(rows, H, V, K, second_only):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(rows + V)
    hid = torch.randn((rows, H), generator=g, device="cuda").to(torch.bfloat16)
    w = (H ** -0.5 * 4 * torch.randn((V, H), generator=g, device="cuda")).to(torch.bfloat16)
    ws = ll.Workspace(int(ll.lib().lilicorr_lm_head_topk_workspace_bytes(rows, H, V, K)))
    want = ll.lm_head_topk(hid, w, K, ws=ws)
    assert ws.status() == 0
    for _ in range(2):
        t0 = time.perf_counter()
        ll.test_lm_head_timeout(hid, w, K, ws, LIMIT, second_only)
        assert ws.status() == TIMEOUT                  # reads and clears it
        dt = time.perf_counter() - t0
        assert dt < 5.0, f"the timed-out call took {dt:.2f} s"
        got = ll.lm_head_topk(hid, w, K, ws=ws)
        assert ws.status() == 0
        assert all(torch.equal(a, b) for a, b in zip(got, want))


def test_lm_head_hook_rejects_other_kernels_and_limits():
    ll = _ll()
    h = torch.zeros((384, 2048), device="cuda", dtype=torch.bfloat16)
    w = torch.zeros((39000, 2048), device="cuda", dtype=torch.bfloat16)
    ws = ll.Workspace(1 << 24)
    for rows, limit in ((16, LIMIT), (100, LIMIT), (384, LIMIT), (256, 10), (256, 10 ** 12)):
        with pytest.raises(ll.LilicorrError):
            ll.test_lm_head_timeout(h[:rows], w, 4, ws, limit)
