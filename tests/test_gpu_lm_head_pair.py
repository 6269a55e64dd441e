"""GPU parity of the fused LM head on pairs of CTAs (more than 128 rows) at the edges of its tiles:
row counts around 128-row halves and 256-row blocks (a CTA with one row, a CTA with none),
vocabularies whose last tile lies half or wholly past the end for one CTA, one step of H and
more steps than stages, the longest candidate lists."""
import numpy as np
import pytest
import torch

from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,H,V,K", [(129, 64, 257, 4), (255, 448, 5000, 8), (256, 128, 384, 32),
                                        (257, 192, 20100, 8), (300, 256, 1000, 1),
                                        (513, 64, 39000, 16), (640, 512, 130, 8)])
def test_pair_lm_head(rows, H, V, K):
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
