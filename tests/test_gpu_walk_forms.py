"""GPU check of the best path over given scores two, four and eight predecessors at a time, also in
a last part round."""
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
