"""Cluster merging against the oracle at the edges of the pair tiles: 256 rows by 128 columns up to
32,768 centres, by 256 beyond."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,terms", [(K, t) for K in (1, 127, 128, 129, 255, 257, 383, 385, 1000)
                                     for t in (1, 2, 3)] + [(32768, 3), (32769, 3)])
def test_merge_matches_oracle(gpu, orc, K, terms):
    rng = np.random.default_rng(K + terms)
    c = rng.random((K, 6)).astype(np.float32)
    c[:, 4] = 1 + 30.0 * rng.random(K) * (rng.random(K) < 0.5)   # half in one group, chains beside it
    c[:, 5] = 1 + 0.3 * rng.random(K)
    if K > 3:
        c[K // 2, 4] = np.nan
    ctx = gpu.Context(0)
    try:
        for eps in (0.0, 0.4 / K, 0.02) if K < 10000 else (0.02,):
            m, n = ctx.merge_clusters(torch.as_tensor(c).cuda(), eps, terms)
            om, on = orc.merge_clusters(c, eps, terms)
            assert n == on and np.array_equal(m, om), eps
    finally:
        ctx.close()
