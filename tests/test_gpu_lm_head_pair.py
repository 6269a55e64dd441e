"""GPU parity of the fused LM head above 128 rows at the edges of its tiles: row counts around 128-row
halves and 256-row blocks (a CTA with one row, a CTA with none), vocabularies whose last tile lies
half or wholly past the end for one CTA, the longest candidate lists; first at short H, one step and
more steps than stages, on single CTAs, then at H from 2048 on, whole steps and a last one of half,
on pairs of CTAs."""
import numpy as np
import pytest
import torch

from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,H,V,K", [(129, 64, 257, 4), (255, 448, 5000, 8), (256, 128, 384, 32),
                                        (257, 192, 20100, 8), (300, 256, 1000, 1),
                                        (513, 64, 39000, 16), (640, 512, 130, 8)])
def test_pair_lm_head(rows, H, V, K):
    _matches_exact(rows, H, V, K)


@pytest.mark.parametrize("rows,H,V,K", [(129, 2048, 257, 4), (255, 2112, 5000, 8),
                                        (256, 2048, 384, 32), (257, 2240, 9000, 8),
                                        (300, 4096, 1000, 1), (513, 2112, 9000, 16),
                                        (640, 2048, 130, 8), (400, 2048, 40000, 16)])
def test_pair_lm_head_long(rows, H, V, K):
    ll = _ll()
    h, w = (torch.zeros((n, H), dtype=torch.bfloat16, device="cuda") for n in (rows, V))
    ws = ll.Workspace(int(ll.lib().lilicorr_lm_head_topk_workspace_bytes(rows, H, V, K)))
    ll.test_lm_head_timeout(h, w, K, ws, 2_000_000)      # refused where no pair takes the call
    assert ws.status() == 6
    _matches_exact(rows, H, V, K)


def _matches_exact(rows, H, V, K):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(rows + V)
    hid = torch.randn((rows, H), generator=g, device="cuda").to(torch.bfloat16)
    w = (H ** -0.5 * 4 * torch.randn((V, H), generator=g, device="cuda")).to(torch.bfloat16)
    ws = ll.Workspace(int(ll.lib().lilicorr_lm_head_topk_workspace_bytes(rows, H, V, K)))
    ids, logp, lse = ll.lm_head_topk(hid, w, K, ws=ws)
    again = ll.lm_head_topk(hid, w, K, ws=ws)
    assert ws.status() == 0
    assert all(torch.equal(a, b) for a, b in zip((ids, logp, lse), again))
    z = hid.double() @ w.double().T
    want, order = torch.sort(z, dim=-1, descending=True, stable=True)
    # fp32 sums of H products of magnitudes whose sum is about 0.64 * 4 * H^0.5
    tol = H * 2.0 ** -23 * 3 * H ** 0.5 + 1e-5
    wl = torch.logsumexp(z, -1)
    assert (lse.double() - wl).abs().max().item() < tol
    assert (logp.double() + lse.double()[:, None] - want[:, :K]).abs().max().item() < tol
    # the ids are the exact ones but for logits closer than the tolerance
    got = torch.gather(z, 1, ids.long())
    assert (got - want[:, :K]).abs().max().item() < 2 * tol
    assert (ids == order[:, :K]).float().mean().item() > 0.99
    assert all(len(set(r)) == K for r in ids.cpu().numpy().tolist())
