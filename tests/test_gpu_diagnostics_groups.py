"""GPU checks of the diagnostics at the edges of their lane groups: score rows of 8, 9, 16, 17
and 32 candidates, paths and runs of more than 32 slots, runs that end on a multiple of 32."""
import numpy as np
import pytest
import torch

from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,K", [(5, 3, 8), (3, 7, 9), (2, 4, 16), (3, 2, 17), (1, 64, 32)])
def test_softmax_and_path_rows(B, L, K):
    ll = _ll()
    rng = np.random.default_rng(K)
    A = rng.uniform(-1, 1, (B, K)).astype(np.float32)
    P = rng.uniform(-1, 1, (B, L - 1, K, K)).astype(np.float32)
    dA, dP = torch.from_numpy(A).cuda(), torch.from_numpy(P).cuda()
    pa, pp = (t.double().cpu() for t in ll.local_softmax(dA, dP, 8.0))
    assert torch.allclose(pa, torch.softmax(8.0 * torch.from_numpy(A).double(), -1), atol=2e-6)
    assert torch.allclose(pp, torch.softmax(8.0 * torch.from_numpy(P).double(), -1), atol=2e-6)
    choice = rng.integers(0, K, (B, L)).astype(np.int32)
    prob, gap, lp = (t.cpu().numpy() for t in ll.path_probs(dA, dP, torch.from_numpy(choice).cuda()))
    for b in range(B):
        z = [8.0 * (A[b] if s == 0 else P[b, s - 1, choice[b, s - 1]]).astype(np.float64)
             for s in range(L)]
        p = np.array([np.exp(r[c] - r.max()) / np.exp(r - r.max()).sum()
                      for r, c in zip(z, choice[b])])
        g = [r[c] - np.delete(r, c).max() for r, c in zip(z, choice[b])]
        assert np.abs(prob[b] - p).max() < 2e-6 and np.abs(gap[b] - g).max() < 1e-5
        # relative error of a probability 1e-6, so of a sum of L logarithms L times that
        assert abs(lp[b] - np.log(p).sum()) < 2e-6 * L + 1e-6 * abs(np.log(p).sum())


@pytest.mark.parametrize("L", [1, 31, 32, 33, 40, 64])
def test_acceptance_runs(L):
    ll = _ll()
    B, K = 12, 3
    rng = np.random.default_rng(L)
    ids = np.argsort(rng.random((B, L, 50)), -1)[..., :K].astype(np.int32)
    truth = ids[..., 1].copy()
    tokens = truth.copy()
    for b in range(1, B):                       # sequence 0 stays right throughout
        tokens[b, rng.integers(0, L)] = 99
        truth[b, (3 * b) % L if b % 2 else L - 1] = 77
    got = [t.cpu().numpy() for t in ll.block_acceptance(
        *(torch.from_numpy(x).cuda() for x in (ids, tokens, truth)))]
    cov = (ids == truth[..., None]).any(-1)

    def run(x):
        return np.where(x.all(1), L, np.argmin(x, 1))
    assert np.array_equal(got[0], cov.astype(np.int32))
    assert np.array_equal(got[1], run(cov)) and np.array_equal(got[2], run(tokens == truth))
