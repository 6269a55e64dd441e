"""GPU check of the record merge where its first-key bound applies (at least K shards, at most
one a thread) and around its limits: exact ids on tied rows, empty and -inf shards, shards
narrower than K."""
import numpy as np
import pytest
import torch

import oracle
from test_gpu_fused import _ll

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,V,K,P", [(3, 4000, 8, 8), (3, 4000, 8, 7), (2, 3000, 1, 256),
                                        (2, 3000, 1, 257), (4, 5000, 16, 152), (2, 600, 32, 200)])
def test_merge_matches_the_whole_row(rows, V, K, P):
    ll = _ll()
    rng = np.random.default_rng(P)
    x = (np.round(rng.standard_normal((rows, V)) * 4) / 4).astype(np.float32)   # many ties
    x[0, : V // 2] = -np.inf                                # whole shards without a finite logit
    cuts = np.linspace(0, V, P + 1).astype(int)
    parts = [ll.topk_lse_partial(torch.from_numpy(x[:, a:b].copy()).cuda(), K, int(a))
             for a, b in zip(cuts[:-1], cuts[1:])]
    ids, logp, lse = ll.topk_lse_merge(torch.stack(parts), K)
    for r in range(rows):
        want, wlogp, wlse = oracle.topk_lse(x[r], K)
        assert np.array_equal(ids[r].cpu().numpy(), want)
        # P fp32 sums added up, each term within an ex2.approx (2^-22)
        assert abs(lse[r].item() - wlse) < 1e-5
        assert np.abs(logp[r].cpu().numpy() - wlogp).max() < 1e-5


@pytest.mark.parametrize("rows,V,K,P", [(3, 4000, 4, 31), (3, 4000, 4, 32), (3, 4000, 3, 152),
                                        (2, 3000, 2, 16), (3, 4000, 8, 15), (3, 4000, 8, 16)])
def test_merge_around_its_bounds_limits(rows, V, K, P):
    test_merge_matches_the_whole_row(rows, V, K, P)
