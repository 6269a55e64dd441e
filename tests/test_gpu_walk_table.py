"""GPU check of the greedy walk along its table of best candidates: ties, infinities and NaN scores,
the largest lattice (scores outside shared memory) and single candidates, with margins."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,K", [(3, 1, 1), (2, 9, 1), (4, 16, 8), (3, 16, 17), (2, 64, 32)])
def test_table_walk(B, L, K):
    ll = _ll()
    rng = np.random.default_rng(K)
    A = np.round(rng.uniform(-1, 1, (B, K)) * 4).astype(np.float32)          # many ties
    P = np.round(rng.uniform(-1, 1, (B, L - 1, K, K)) * 4).astype(np.float32)
    P[0, L // 2:, :, 0] = -np.inf
    if L > 2:
        P[-1, 1] = np.inf                                  # a slot pair of equal infinities
    ids = rng.integers(0, 1000, (B, L, K)).astype(np.int32)
    choice, tokens, margin = (t.cpu().numpy() for t in ll.greedy_walk(
        *(torch.from_numpy(x).cuda() for x in (A, P, ids))))
    for b in range(B):
        c = oracle.greedy_walk(A[b], P[b])[0]
        assert np.array_equal(choice[b], c)
        assert np.array_equal(tokens[b], ids[b, np.arange(L), c])
        for s in range(L):
            row = (A[b] if s == 0 else P[b, s - 1, c[s - 1]]).astype(np.float32)
            rest = np.delete(row, c[s])
            want = row[c[s]] - rest.max() if K > 1 else np.inf
            assert margin[b, s] == want or (np.isnan(want) and np.isnan(margin[b, s]))


def test_nan_scores_choose_a_candidate():
    ll = _ll()
    A = torch.full((2, 5), float("nan"), device="cuda")
    P = torch.zeros((2, 3, 5, 5), device="cuda")
    P[:, 1] = float("nan")
    P[1, 0, 0, 3] = 1.0
    ids = torch.arange(2 * 4 * 5, dtype=torch.int32, device="cuda").view(2, 4, 5)
    choice, tokens, _ = ll.greedy_walk(A, P, ids)
    assert choice.cpu().tolist() == [[0, 0, 0, 0], [0, 3, 0, 0]]
    assert torch.equal(tokens, torch.gather(ids, 2, choice[..., None].long())[..., 0])
