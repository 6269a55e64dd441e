"""GPU check of the pair scores where several groups of lanes share a block of outputs, from
sixteen (one candidate) down to one (13 to 16 candidates), against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,K,d", [(2, 3, 1, 4), (2, 3, 4, 2048), (3, 4, 5, 132), (2, 5, 8, 1024),
                                     (2, 3, 9, 516), (2, 3, 12, 64), (3, 3, 16, 512)])
def test_pair_scores_shared_columns(B, L, K, d):
    ll = _ll()
    rng = np.random.default_rng(d + K)
    out, inn = (rng.standard_normal((B, L, K, d)).astype(np.float32) for _ in range(2))
    anc = rng.standard_normal((B, d)).astype(np.float32)
    A, P = (t.cpu().numpy() for t in ll.pair_scores(*(torch.from_numpy(x).cuda()
                                                      for x in (out, inn, anc))))
    for b in range(B):
        wa, wp = oracle.pair_scores(out[b], inn[b], anc[b])
        # fp32 sums of d terms over norms of about d: d 2^-24 / sqrt(d), and the divisions
        tol = 2.0 ** -24 * (d ** 0.5 + 8) * 2
        assert np.abs(A[b] - wa).max() <= tol and np.abs(P[b] - wp).max() <= tol
