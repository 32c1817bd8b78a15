"""Clustering parity with the oracle where the candidate scans and the packed sums have edges: equal
distances everywhere (a constant field and constant attributes), weights the approximate scan does
not cover, one cell, more cells than voxels along an axis, rows around a tile's width, 2D + time."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEFAULT = dict(w_p=1.0, w_f=1.0, w_d=0.05, c_f=1.0, eps_c=0.0, max_iter=4)


@pytest.mark.parametrize("nx,ny,nz,T,P,k,kw,data", [
    (24, 20, 12, 6, 9000, (3, 3, 2, 2), {}, "noise"),
    (24, 20, 12, 6, 9000, (3, 3, 2, 2), {}, "constant"),
    (24, 20, 12, 6, 9000, (3, 3, 2, 2), dict(w_f=0.0, w_p=0.0), "noise"),
    (24, 20, 12, 6, 9000, (3, 3, 2, 2), dict(w_d=0.0), "noise"),
    (24, 20, 12, 6, 5000, (3, 2, 2, 3), dict(w_d=-0.5), "noise"),
    (24, 20, 12, 6, 5000, (2, 2, 2, 3), dict(c_f=0.0), "noise"),
    (33, 9, 5, 3, 20000, (1, 1, 1, 1), {}, "noise"),
    (9, 5, 3, 4, 700, (9, 5, 3, 4), {}, "noise"),
    (6, 5, 3, 4, 700, (12, 10, 6, 8), {}, "noise"),
    (65, 37, 1, 9, 4000, (5, 4, 1, 3), {}, "steps"),
    (40, 24, 9, 5, 3000, (5, 3, 2, 1), dict(w_f=20.0, w_p=20.0, w_d=0.01), "steps"),
    (17, 13, 11, 5, 0, (2, 3, 2, 2), {}, "noise")])
def test_clustering_matches_oracle(gpu, orc, nx, ny, nz, T, P, k, kw, data):
    rng = np.random.default_rng(nx * 100 + P)
    f = rng.normal(1.0, 0.3, size=(T, nz, ny, nx)).astype(np.float32)
    pos = (rng.random((T, 3, P)) * (1.01 * np.array([nx, ny, nz]))[None, :, None]).astype(np.float32)
    a = rng.normal(0.5, 0.2, size=(T, 1, P)).astype(np.float32)
    if data == "constant":
        f[:], a[:] = 0.25, 0.5
        pos = np.floor(pos * 2) / 2          # many equal positions
    elif data == "steps":
        f = np.round(f * 2) / 2
        a = np.round(a * 4) / 4
    f[0, 0, 0, 0] = np.nan
    p = dict(DEFAULT, **kw)
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x.astype(np.float32)).cuda().contiguous() for x in (f, pos, a)))
        ctx.bin()
        fl, pl, c, n, it = ctx.cluster(0, T, 0, k, **p)
        key = ctx.bins("cpu")[0].numpy()
    finally:
        ctx.close()
    o = orc.slic(f, pos.astype(np.float32), a, key, 0, T, 0, k, **p)
    assert it == o[4]
    assert np.array_equal(fl.cpu().numpy(), o[0])
    assert np.array_equal(pl.cpu().numpy(), o[1])
    assert np.array_equal(n, o[3])
    assert np.array_equal(c.view(np.uint32), o[2].view(np.uint32))
