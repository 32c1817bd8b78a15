"""Where one block ranks the features: windows of up to 12,288 words of label bits and 8192 features.
Beyond either limit the ranks are a chain of passes over the whole GPU, and both give the oracle's
statistics."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,T,members,one_block", [
    (64, 64, 32, 3, 8192, True), (64, 64, 32, 3, 8193, False), (64, 64, 32, 3, 200000, False),
    (64, 64, 49, 2, 100, False), (33, 31, 7, 4, 5000, True), (96, 64, 64, 4, 31542, False)])
def test_ranks_at_the_limits(gpu, orc, nx, ny, nz, T, members, one_block):
    rng = np.random.default_rng(members)
    n = T * nz * ny * nx
    f = np.full(n, -1.0, np.float32)
    f[rng.permutation(n)[:members]] = 1 + rng.random(members).astype(np.float32)
    f = f.reshape(T, nz, ny, nx)
    pos = (rng.random((T, 3, 500)) * np.array([nx, ny, nz])[None, :, None]).astype(np.float32)
    a = rng.random((T, 1, 500)).astype(np.float32)
    preds = [(0, 0, 0, 0.0, 0.0)]
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x).cuda().contiguous() for x in (f, pos, a)))
        ctx.bin()
        lab, k = ctx.segment(0, T, preds, 0)  # no edges: every member is a feature
        ctx.profiling(True)
        ctx.kernel_times(True)
        g = ctx.features(0, T, lab, preds, 0)
        names = set(ctx.kernel_times(True))
    finally:
        ctx.close()
    assert ("k_feat_ranks" in names) == one_block and ("k_comp_fid" in names) != one_block
    b, olab, on, o = orc.run_all(f, pos, a, 0, T, preds, 0)
    assert k == on == members == len(g)
    for key in ("label", "n_vox", "n_pts"):
        assert np.array_equal(g[key], o[key]), key
    assert np.array_equal(np.concatenate([g["bbox_min"], g["bbox_max"]], 1), o["bbox"])
    assert np.array_equal(g["sumq"][:, :1], o["sumq"][:, :1])
    assert np.array_equal(g["sum_field"], f[f > 0].astype(np.float64))


@pytest.mark.parametrize("members,A", [(4095, 2), (4096, 1), (4097, 2), (20011, 8), (65537, 3),
                                       (140001, 2), (524289, 1)])
def test_records_by_copy_and_by_feature(gpu, members, A):
    """Single-voxel features around the numbers where a lane sums one copy, or all copies, of a
    feature: 16 copies and 65,536 in all, then fewer copies, then one. Each has one sample."""
    T, nx, ny, nz = 3, 96, 64, 32
    rng = np.random.default_rng(members)
    n = T * nz * ny * nx
    at = np.sort(rng.permutation(n)[:members])
    f = np.full(n, -1.0, np.float32)
    f[at] = 1 + rng.random(members).astype(np.float32)
    t, v = at // (n // T), at % (n // T)
    P = int(np.bincount(t, minlength=T).max())
    pos = np.full((T, 3, P), -5.0, np.float32)       # outside, but for one point per member
    a = np.zeros((T, A, P), np.float32)
    k = np.arange(members) - np.searchsorted(t, np.arange(T))[t]
    xyz = np.stack([v % nx, v // nx % ny, v // (nx * ny)])
    pos[t, :, k] = (xyz + 0.5).T
    a[t, :, k] = 1 + rng.integers(0, 1 << 20, (members, A)).astype(np.float32) / (1 << 20)
    preds = [(0, 0, 0, 0.0, 0.0)]
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x).cuda().contiguous()
                   for x in (f.reshape(T, nz, ny, nx), pos, a)))
        ctx.bin()
        lab, m = ctx.segment(0, T, preds, 0)
        g = [ctx.features(0, T, lab, preds, 0), ctx.features(0, T, lab.clone(), preds, 0)]
    finally:
        ctx.close()
    for r in g:
        assert m == len(r) == members and np.array_equal(r["label"], at)
        assert (r["n_vox"] == 1).all() and (r["n_pts"] == 1).all()
        assert np.array_equal(r["mean_attr"][:, :A], a[t, :, k].astype(np.float64))
        assert (r["std_attr"][:, :A] == 0).all() and (r["std_field"] == 0).all()
        assert np.array_equal(r["sum_field"], f[at].astype(np.float64))
        assert np.array_equal(r["min_field"], f[at]) and np.array_equal(r["max_field"], f[at])
        c = np.stack([t, *xyz[::-1]], 1)
        assert np.array_equal(r["centroid"], c.astype(np.float64))
        assert np.array_equal(r["bbox_min"], c) and np.array_equal(r["bbox_max"], c)
