"""The sums of squares behind a feature's deviations: which samples are rounded together, and how far
the rounding may move a deviation.

The point statistics walk windows of 256 records of a field step, and round the squares that a
feature's samples have in one pack of at most 32 of a window's members together. Records are grouped
by buckets of 2048 consecutive voxels, in any order inside a bucket: the cases fill whole buckets
with whole windows, so that which samples can meet follows from their buckets alone."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SPATIAL, FIELD, GT = 1, 0, 0


def _features(gpu, field, pos, attr, field_step=None):
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x).cuda().contiguous() for x in (field, pos, attr)),
                 field_step=field_step)
        ctx.bin()
        preds = [(FIELD, 0, GT, 0.0, 0.0)]
        lab, n = ctx.segment(0, field.shape[0], preds, SPATIAL)
        f = ctx.features(0, field.shape[0], lab, preds, SPATIAL)
    finally:
        ctx.close()
    assert n == len(f)
    return f


@pytest.mark.parametrize("A", [1, 4, 8])
def test_samples_of_two_windows_are_rounded_apart(gpu, A):
    """Every feature is a column of two voxels with one sample each, in two buckets (planes of 2048
    voxels) of 1024 records: the samples lie in different windows. A square has at most 48 bits and
    the sum of two 53, so nothing is rounded, and the deviation is exactly half their difference."""
    T, nx, ny, nz, P = 64, 32, 64, 8, 40960
    field = np.full((T, nz, ny, nx), -1.0, np.float32)
    field[:, :2, ::8, ::2] = 1.0
    x, y = np.meshgrid(np.arange(0, nx, 2), np.arange(0, ny, 8))
    x, y = x.ravel(), y.ravel()                     # 128 columns
    rng = np.random.default_rng(A)
    p = np.empty((3, P), np.float32)
    for z in range(2):                              # 128 members and 896 others in each plane
        i = 1024 * z
        p[:, i:i + 128] = np.stack([x, y, np.full(128, z)])
        p[:, i + 128:i + 1024] = np.stack([rng.integers(0, 16, 896) * 2 + 1,
                                           rng.integers(0, ny, 896), np.full(896, z)])
    rest = P - 2048                                 # the rest of the step, so that blocks are long
    p[:, 2048:] = np.stack([rng.integers(0, nx, rest), rng.integers(0, ny, rest),
                            rng.integers(2, nz, rest)])
    pos = np.tile(p + 0.5, (T, 1, 1))
    attr = (1.0 + rng.random((T, A, P))).astype(np.float32)
    attr[:, :, 1024:1152] = attr[:, :, :128] * (1 + 1e-5 * rng.standard_normal((T, A, 128)))
    f = _features(gpu, field, pos, attr)
    assert len(f) == 128 * T and (f["n_vox"] == 2).all() and (f["n_pts"] == 2).all()
    # features come by label: step, then the column (y, x) of the lower plane
    a, b = (attr[:, :, i:i + 128].astype(np.float64).transpose(0, 2, 1).reshape(-1, A)
            for i in (0, 1024))
    assert np.array_equal(f["std_attr"][:, :A], np.abs(a - b) / 2)


@pytest.mark.parametrize("n", [3, 4, 7, 24, 32])
@pytest.mark.parametrize("spread", [0.0, 1e-7, 1e-6, 1e-4])
def test_nearly_equal_samples(gpu, n, spread):
    """Features of one voxel with n samples that are equal or nearly so. A pack's sum of squares
    keeps 48 bits, the sums and the mean's square 53: the variance is off by no more than 2^-47 of
    the mean's square from the former and 2^-50 from the latter, and a negative one counts as zero."""
    nx = 64
    field = np.full((1, nx, nx, nx), -1.0, np.float32)
    field[0, ::4, ::4, ::4] = 1.0
    c = np.arange(0, nx, 4)
    z, y, x = (g.ravel() for g in np.meshgrid(c, c, c, indexing="ij"))
    rng = np.random.default_rng(n)
    order = rng.permutation(np.repeat(np.arange(x.size), n))
    pos = (np.stack([x, y, z])[:, order] + 0.5).astype(np.float32)[None]
    base = 300.0 + 1700.0 * rng.random(x.size)
    attr = (base[order] * (1 + spread * rng.standard_normal(order.size))).astype(np.float32)
    f = _features(gpu, field, pos, attr[None, None])
    assert len(f) == x.size and (f["n_pts"] == n).all()
    v = np.empty((x.size, n))
    v[order[np.argsort(order, kind="stable")], np.tile(np.arange(n), x.size)] = \
        attr[np.argsort(order, kind="stable")]
    m = v.mean(1)
    var = ((v - m[:, None]) ** 2).mean(1)
    bound = (2.0 ** -47 + 2.0 ** -50) * m * m
    assert (np.abs(f["std_attr"][:, 0] ** 2 - var) <= bound).all()


@pytest.mark.parametrize("nx,P,M,r,T,least", [(32, 20000, 300, 4, 8, 0.08),
                                              (48, 30000, 300, 2, 8, 0.10)])
def test_samples_of_one_point_lie_close(gpu, nx, P, M, r, T, least):
    """All point steps of a field step are placed at the same time, each in the order of its points,
    so the r samples of a point lie close together in their bucket and often share a pack: in 25 to
    30 (r = 4) and 21 to 24 per cent (r = 2) of these features of one resting point the rounding of
    two or more samples together shows. (With every block's samples sorted by bucket before they are
    stored it is 0.4 and 6 per cent, and the deviations are other ones.)"""
    rng = np.random.default_rng(nx)
    field = np.full((T, nx, nx, nx), -1.0, np.float32)
    even = np.arange(0, nx, 2)
    z, y, x = (even[c] for c in np.unravel_index(rng.permutation(even.size ** 3)[:M],
                                                 (even.size,) * 3))
    field[:, z, y, x] = 1.0
    who = rng.permutation(P)
    p = np.empty((3, P))
    p[:, who[:M]] = np.stack([x, y, z])
    p[:, who[M:]] = rng.integers(0, nx, (3, P - M))
    p[0, who[M:]] = p[0, who[M:]] // 2 * 2 + 1      # no member there
    pos = np.tile((p + 0.5).astype(np.float32), (T * r, 1, 1))
    attr = ((1 + rng.random(P)) * (1 + 1e-5 * rng.standard_normal((T * r, P)))).astype(np.float32)
    f = _features(gpu, field, pos, attr[:, None], [j // r for j in range(T * r)])
    assert len(f) == M * T and (f["n_pts"] == r).all()
    v = attr[:, who[:M][np.argsort((z * nx + y) * nx + x)]].astype(np.float64)
    v = v.reshape(T, r, M).transpose(0, 2, 1).reshape(-1, r)
    exact = np.sqrt(np.maximum((v * v).sum(1) / r - (v.sum(1) / r) ** 2, 0.0))
    assert (f["std_attr"][:, 0] != exact).mean() >= least
