"""Per-cluster summaries at the sizes where the run and table arithmetic can go wrong: one label
everywhere (every run of a block meets in one place), more labels than a block's table holds,
windows of one step, row lengths around a block, few samples."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,T,P,K,lab", [
    (1, 1, 1, 1, 1, 1, "one"), (33, 5, 3, 2, 300, 3, "one"), (64, 64, 16, 17, 70000, 2, "most"),
    (300, 40, 9, 3, 2000, 5000, "random"), (129, 64, 20, 4, 30000, 9000, "blocks"),
    (1100, 90, 1, 5, 5000, 40, "most"), (5, 200, 30, 18, 1000, 700, "random")])
def test_summaries_match_oracle(gpu, orc, nx, ny, nz, T, P, K, lab):
    rng = np.random.default_rng(nx + K)
    f = rng.normal(1.0, 2.0, size=(T, nz, ny, nx)).astype(np.float32)
    pos = (rng.random((T, 3, P)) * (1.02 * np.array([nx, ny, nz]))[None, :, None]).astype(np.float32)
    a = rng.lognormal(size=(T, 1, P)).astype(np.float32)
    f.reshape(-1)[::1001] = np.inf
    fl = rng.integers(-1, K, size=f.shape).astype(np.int32)
    pl = rng.integers(-1, K, size=(T, P)).astype(np.int32)
    if lab == "one":
        fl[:], pl[:] = 0, 0
    elif lab == "most":
        fl[rng.random(f.shape) < 0.9] = 1
        pl[rng.random(pl.shape) < 0.9] = 1
    elif lab == "blocks":  # small cells, as a clustering leaves them
        i = np.indices(f.shape)
        fl[:] = ((i[1] // 4 * 16 + i[2] // 4) * 33 + i[3] // 4) % K
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x).cuda().contiguous() for x in (f, pos, a)))
        ctx.bin()
        g = ctx.cluster_stats(0, T, 0, torch.as_tensor(fl).cuda(), torch.as_tensor(pl).cuda(), K)
        key = ctx.bins("cpu")[0].numpy()
    finally:
        ctx.close()
    o = orc.cluster_stats(f, pos, a, key, 0, T, 0, fl, pl, K)
    for k in ("n_field", "n_point", "lo", "hi"):
        assert np.array_equal(g[k], o[k]), k
    for k in ("mean_field", "mean_point"):
        assert np.array_equal(g[k], o[k], equal_nan=True), k
    for k in ("std_field", "std_point"):  # fp64 sums in no fixed order
        np.testing.assert_allclose(g[k], o[k], rtol=1e-9, atol=1e-12, equal_nan=True)
