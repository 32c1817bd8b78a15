"""Clustering parity with the oracle where a tile's four steps reach more cells than a block lists, so
that it takes two steps at a time, or one: cells of a step or two, few voxels wide."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,T,k", [
    (24, 20, 12, 8, (6, 5, 3, 8)), (24, 20, 12, 7, (6, 5, 3, 7)), (24, 20, 12, 6, (6, 5, 3, 6)),
    (16, 16, 8, 9, (5, 5, 2, 9)), (17, 16, 12, 5, (6, 4, 4, 10)), (24, 24, 8, 4, (8, 8, 2, 4)),
    (40, 40, 1, 9, (13, 13, 1, 9)), (48, 33, 1, 6, (24, 16, 1, 6))])
@pytest.mark.parametrize("kw", [{}, dict(w_d=1.0), dict(w_f=0.0, w_p=2.0)])
def test_small_time_cells(gpu, orc, nx, ny, nz, T, k, kw):
    rng = np.random.default_rng(nx + T + k[0])
    P = 3000
    f = rng.normal(1.0, 0.3, size=(T, nz, ny, nx)).astype(np.float32)
    pos = (rng.random((T, 3, P)) * np.array([nx, ny, nz])[None, :, None]).astype(np.float32)
    a = rng.normal(0.5, 0.2, size=(T, 1, P)).astype(np.float32)
    p = dict(dict(w_p=1.0, w_f=1.0, w_d=0.05, c_f=1.0, eps_c=0.0, max_iter=4), **kw)
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x).cuda().contiguous() for x in (f, pos, a)))
        ctx.bin()
        fl, pl, c, n, it = ctx.cluster(0, T, 0, k, **p)
        key = ctx.bins("cpu")[0].numpy()
    finally:
        ctx.close()
    o = orc.slic(f, pos, a, key, 0, T, 0, k, **p)
    assert it == o[4]
    assert np.array_equal(fl.cpu().numpy(), o[0]) and np.array_equal(pl.cpu().numpy(), o[1])
    assert np.array_equal(n, o[3]) and np.array_equal(c.view(np.uint32), o[2].view(np.uint32))
