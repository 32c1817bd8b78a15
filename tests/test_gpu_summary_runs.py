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


@pytest.mark.parametrize("n", [1, 3, 4, 5, 1027, 300001])
@pytest.mark.parametrize("shift", [0, 1, 2])  # labels that start off a 16-byte boundary
def test_relabel_matches_numpy(gpu, n, shift):
    rng = np.random.default_rng(n + shift)
    K = 77
    lab = rng.integers(-2, K, size=n + shift).astype(np.int32)
    m = rng.permutation(K).astype(np.int32)
    ctx = gpu.Context(0)
    try:
        d = torch.as_tensor(lab).cuda()
        ctx.relabel(d[shift:], torch.as_tensor(m).cuda())
        want = lab.copy()
        want[shift:] = np.where(lab[shift:] >= 0, m[np.maximum(lab[shift:], 0)], lab[shift:])
        assert np.array_equal(d.cpu().numpy(), want)
        for at in {0, n // 2, n - 1}:  # one label out of range anywhere: nothing changes
            bad = torch.as_tensor(lab).cuda()
            bad[shift + at] = K
            before = bad.clone()
            with pytest.raises(gpu.MsfError) as e:
                ctx.relabel(bad[shift:], torch.as_tensor(m).cuda())
            assert e.value.status == gpu.MSF_ERR_INVALID_ARG
            assert torch.equal(bad, before)
    finally:
        ctx.close()


@pytest.mark.parametrize("K", [2, 256, 257, 700, 5000])
def test_merge_chains_match_oracle(gpu, orc, K):
    """Chains of matches that cross the pair tiles, groups interleaved by index."""
    rng = np.random.default_rng(K)
    c = np.zeros((K, 6), np.float32)
    g = rng.integers(0, 5, K)
    c[:, 4] = (10.0 ** g) * (1 + 0.004 * rng.permutation(K) / K * 40)
    c[:, 5] = 1.0
    ctx = gpu.Context(0)
    try:
        m, n = ctx.merge_clusters(torch.as_tensor(c).cuda(), 0.002)
    finally:
        ctx.close()
    om, on = orc.merge_clusters(c, 0.002, 3)
    assert n == on and np.array_equal(m, om)
