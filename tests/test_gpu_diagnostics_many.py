"""GPU checks of the diagnostics of many sequences: paths by a warp each beside paths by a CTA each
(numbers that leave a last CTA part empty), and runs by four lanes each beside runs by a warp."""
import pytest
import torch

from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,K", [(3, 1, 5), (1221, 1, 32), (1221, 2, 32), (1221, 3, 8),
                                   (4563, 9, 4), (4563, 10, 4)])
def test_paths(B, L, K):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(B + L)
    A = torch.randn(B, K, generator=g, device="cuda")
    P = torch.randn(B, L - 1, K, K, generator=g, device="cuda")
    choice = torch.randint(0, K, (B, L), generator=g, device="cuda", dtype=torch.int32)
    choice[-1, L // 2] = K                         # not a candidate: no probability there
    prob, gap, lp = ll.path_probs(A, P, choice, 2.0)
    at = choice.long().clamp(max=K - 1)
    z = torch.cat([A[:, None], P.gather(2, at[:, :-1, None, None].expand(-1, -1, 1, K))[:, :, 0]], 1)
    z = 2.0 * z.double()
    lse = torch.logsumexp(z, -1)
    zc = z.gather(2, at[..., None])[..., 0]
    other = z.scatter(2, at[..., None], -float("inf")).amax(-1)
    ok = torch.ones_like(choice, dtype=torch.bool)
    ok[-1, L // 2:L // 2 + 2] = False
    assert torch.isnan(prob[~ok]).all() and torch.isnan(gap[~ok]).all() and torch.isnan(lp[-1])
    assert ((prob.double() - (zc - lse).exp()).abs()[ok] < 2e-6).all()
    assert ((gap.double() - (zc - other)).abs()[ok] < 1e-5).all()
    want = (zc - lse).sum(1)[:-1]
    # relative error of a probability 1e-6, so of a sum of L logarithms L times that
    assert ((lp[:-1].double() - want).abs() < 2e-6 * L + 1e-6 * want.abs()).all()


@pytest.mark.parametrize("B,L,K", [(4869, 1, 4), (4869, 3, 1), (4869, 4, 32), (4869, 5, 2),
                                   (4869, 8, 3), (4869, 9, 3), (4863, 4, 2)])
def test_runs(B, L, K):
    ll = _ll()
    g = torch.Generator(device="cuda").manual_seed(L)
    ids = torch.randint(0, 2 * K + 1, (B, L, K), generator=g, device="cuda", dtype=torch.int32)
    truth = torch.randint(0, 2 * K + 1, (B, L), generator=g, device="cuda", dtype=torch.int32)
    truth[::5] = ids[::5, :, -1]                   # every fifth covered throughout
    tokens = torch.where(torch.rand(B, L, generator=g, device="cuda") < 0.8, truth, truth + 1)
    covered, prefix, accepted = ll.block_acceptance(ids, tokens, truth)
    cov, same = (ids == truth[..., None]).any(-1), tokens == truth
    assert torch.equal(covered, cov.int())
    assert torch.equal(prefix, cov.int().cumprod(1).sum(1).int())
    assert torch.equal(accepted, same.int().cumprod(1).sum(1).int())
