"""Clustering parity with the oracle where the approximate scan is least sure of the best: values
that differ widely or not at all between centres, weights at and beyond what the scan's error bound
covers (odd lists of centres, clipped warps and steps)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DEFAULT = dict(w_p=1.0, w_f=1.0, w_d=0.05, c_f=1.0, eps_c=0.0, max_iter=4)


@pytest.mark.parametrize("nx,ny,nz,T,P,k,kw,data", [
    (48, 40, 24, 9, 9000, (6, 5, 3, 3), dict(w_d=1.0), "smooth"),
    (48, 40, 24, 9, 9000, (6, 5, 3, 3), dict(w_d=1.0), "constant"),
    (47, 33, 9, 7, 9000, (6, 4, 2, 3), dict(w_d=50.0), "noise"),
    (33, 17, 5, 3, 4000, (8, 4, 2, 2), dict(w_f=0.0, w_p=0.0, w_d=3.0), "noise"),
    (32, 16, 8, 4, 4000, (4, 2, 1, 1), dict(w_d=1e-8), "steps"),
    (32, 16, 8, 4, 4000, (4, 2, 1, 2), dict(w_f=1e-12, w_p=1e-12), "noise"),
    (32, 16, 8, 4, 4000, (4, 2, 1, 2), dict(w_f=1e10, w_p=1e10), "noise"),
    (40, 40, 1, 8, 4000, (5, 5, 1, 2), dict(w_d=0.5, c_f=8.0), "smooth")])
def test_clustering_matches_oracle(gpu, orc, nx, ny, nz, T, P, k, kw, data):
    rng = np.random.default_rng(nx * 100 + T)
    f = rng.normal(1.0, 0.3, size=(T, nz, ny, nx)).astype(np.float32)
    pos = (rng.random((T, 3, P)) * (1.01 * np.array([nx, ny, nz]))[None, :, None]).astype(np.float32)
    a = rng.normal(0.5, 0.2, size=(T, 1, P)).astype(np.float32)
    if data == "constant":
        f[:], a[:] = 0.25, 0.5
        pos = np.floor(pos * 2) / 2          # many equal positions
    elif data == "steps":
        f = np.round(f * 2) / 2
        a = np.round(a * 4) / 4
    elif data == "smooth":
        i = np.indices(f.shape)
        f = np.sin(i[3] / 9.0) + np.cos(i[2] / 7.0) + 0.1 * i[1] + 0.05 * i[0]
        a[:, 0] = np.sin(pos[:, 0] / 9.0) + 0.1 * pos[:, 2]
    p = dict(DEFAULT, **kw)
    f, pos, a = (x.astype(np.float32) for x in (f, pos, a))
    f[0, 0, 0, 0] = np.nan
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x).cuda().contiguous() for x in (f, pos, a)))
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
