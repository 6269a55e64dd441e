"""GPU checks of the walks over given scores in each form they take: the greedy walk step by step
(one and two slots; few slots of many candidates in many sequences) and along its table (rows of 16
and 32 scores from different candidates, other sizes from the first), with ties, infinities and NaN
scores, and the best path two, four and eight predecessors at a time, also in a last part round."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu


def _scores(B, L, K, rng):
    A = np.round(rng.uniform(-1, 1, (B, K)) * 4).astype(np.float32)          # many ties
    P = np.round(rng.uniform(-1, 1, (B, L - 1, K, K)) * 4).astype(np.float32)
    return A, P, rng.integers(0, 1000, (B, L, K)).astype(np.int32)


def _rows(x):
    """Rows as the walk reads them: a NaN in front is chosen, any other never."""
    front = np.isnan(x[..., :1])
    x = np.where(np.isnan(x), -np.inf, x)
    x[..., :1] = np.where(front, np.inf, x[..., :1])
    x[..., 1:] = np.where(front, -np.inf, x[..., 1:])
    return x


@pytest.mark.parametrize("B,L,K", [
    (3, 1, 1), (3, 1, 31), (5, 2, 3), (4, 2, 32), (4, 3, 16), (4, 8, 32), (3, 20, 24),
    (700, 2, 7), (700, 3, 9), (700, 5, 16), (700, 6, 16), (650, 8, 24), (620, 10, 32), (620, 11, 32)])
def test_greedy_walk(B, L, K):
    ll = _ll()
    rng = np.random.default_rng(B + 64 * L + K)
    A, P, ids = _scores(B, L, K, rng)
    A[0] = -np.inf
    A[1, rng.integers(0, K)] = np.nan
    A[2, 0] = np.nan
    if L > 1:
        P[::3, 0][rng.random(P[::3, 0].shape) < 0.3] = np.nan
        P[1::3, L // 2 - 1] = -np.inf
        P[1::3, L // 2 - 1][rng.random(P[1::3, 0].shape) < 0.5] = np.nan
        P[2::3, -1, :, K // 2:] = np.inf
    choice, tokens, _ = (t.cpu().numpy() for t in ll.greedy_walk(
        *(torch.from_numpy(x).cuda() for x in (A, P, ids))))
    A, P = _rows(A), _rows(P)
    for b in range(B):
        c = oracle.greedy_walk(A[b], P[b])[0]
        assert np.array_equal(choice[b], c), b
        assert np.array_equal(tokens[b], ids[b, np.arange(L), c])


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 8, 9, 12, 13, 20, 28, 31])
def test_best_path(K):
    ll = _ll()
    B, L = 4, 11
    A, P, ids = _scores(B, L, K, np.random.default_rng(K))
    choice, tokens, score = (t.cpu().numpy() for t in ll.best_path(
        *(torch.from_numpy(x).cuda() for x in (A, P, ids)), 2.0))
    for b in range(B):
        c, g = oracle.viterbi(A[b].astype(np.float64), P[b].astype(np.float64), 2.0)
        assert np.array_equal(choice[b], c) and score[b] == g       # whole numbers: exact
        assert np.array_equal(tokens[b], ids[b, np.arange(L), c])
