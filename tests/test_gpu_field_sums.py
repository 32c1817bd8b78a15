"""The sums behind a feature's field statistics keep fp64: features of nearly equal field values."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dx,dy,dz", [(1, 2, 1), (1, 1, 2), (1, 2, 4), (2, 2, 2), (1, 4, 3),
                                      (3, 3, 3), (7, 3, 3)])
@pytest.mark.parametrize("spread", [1e-7, 1e-5])
def test_deviation_of_nearly_equal_values(gpu, dx, dy, dz, spread):
    """A square has 48 bits, so two voxels' sums are exact. More: a thread adds up to 8 voxels, a
    warp one or two a lane in five steps, and the tiles a feature crosses (up to eight) add in
    memory; the quotients and the mean's square round four times. 16 roundings of 2^-53 of the
    mean's square bound the variance's error (two voxels: the four)."""
    n, step = 64, 8
    c = np.arange(0, n, step)
    field = np.full((1, n, n, n), -1.0, np.float32)
    rng = np.random.default_rng(dx + 10 * dy + 100 * dz)
    blocks = np.abs(1 + rng.random((c.size,) * 3))[..., None, None, None] * (
        1 + spread * rng.standard_normal((c.size,) * 3 + (dz, dy, dx)))
    blocks = blocks.astype(np.float32)
    for i, z in enumerate(c):
        for j, y in enumerate(c):
            for k, x in enumerate(c):
                field[0, z:z + dz, y:y + dy, x:x + dx] = blocks[i, j, k]
    pos, attr = torch.full((1, 3, 1), 0.5), torch.ones((1, 1, 1))
    ctx = gpu.Context(0)
    try:
        ctx.load(torch.as_tensor(field).cuda(), pos.cuda(), attr.cuda())
        ctx.bin()
        preds = [(0, 0, 0, 0.0, 0.0)]
        lab, m = ctx.segment(0, 1, preds, 1)
        f = ctx.features(0, 1, lab, preds, 1)
    finally:
        ctx.close()
    v = blocks.astype(np.float64).reshape(c.size ** 3, -1)
    assert m == len(f) == len(v) and (f["n_vox"] == dx * dy * dz).all()
    mean = v.mean(1)
    var = ((v - mean[:, None]) ** 2).mean(1)
    bound = (4 if v.shape[1] == 2 else 16) * 2.0 ** -53 * mean * mean
    np.testing.assert_allclose(f["mean_field"], mean, rtol=16 * 2.0 ** -53)
    assert (np.abs(f["std_field"] ** 2 - var) <= bound).all()


def test_centroids_are_ieee_quotients(gpu):
    """Centroids are the exact integer sums of the coordinates over the voxel count, rounded once:
    feature sizes from one voxel to some thousands, on rows of up to 4096 voxels."""
    rng = np.random.default_rng(3)
    T, ny, nx = 9, 64, 4096
    f = np.where(rng.random((T, 1, ny, nx)) < 0.45, 1.0, -1.0).astype(np.float32)
    ctx = gpu.Context(0)
    try:
        ctx.load(torch.as_tensor(f).cuda(), torch.full((T, 3, 1), 0.5).cuda(),
                 torch.ones((T, 1, 1)).cuda())
        ctx.bin()
        preds = [(0, 0, 0, 0.0, 0.0)]
        for edges in (1, 2):
            lab, n = ctx.segment(0, T, preds, edges)
            g = ctx.features(0, T, lab, preds, edges)
            l = lab.cpu().numpy().ravel()
            at = np.flatnonzero(l >= 0)
            which = np.searchsorted(g["label"], l[at])
            count = np.bincount(which, minlength=n)
            assert np.array_equal(count, g["n_vox"])
            c = np.stack(np.unravel_index(at, (T, 1, ny, nx)), 1)
            for j in range(4):
                s = np.zeros(n, np.int64)
                np.add.at(s, which, c[:, j])
                assert np.array_equal(g["centroid"][:, j], s / count), j
    finally:
        ctx.close()
