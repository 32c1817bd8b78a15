"""Labels and features against the oracle for windows on both sides of the line below which the
joins, and the voxel and point statistics, go out as one launch; with empty tiles between."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,T,A,edges,mask", [
    (5, 3, 2, 2, 1, 7, "all"), (33, 17, 9, 1, 1, 7, "half"), (32, 32, 32, 8, 2, 7, "one"),
    (32, 32, 32, 8, 3, 6, "none"), (64, 64, 64, 14, 1, 7, "slab"), (64, 64, 64, 20, 7, 7, "slab"),
    (64, 64, 64, 14, 2, 5, "half"), (64, 64, 64, 14, 1, 4, "half")])
def test_windows_match_oracle(gpu, orc, nx, ny, nz, T, A, edges, mask):
    rng = np.random.default_rng(nx + 7 * T + A)
    shape = (T, nz, ny, nx)
    on = np.zeros(shape, bool)
    if mask == "all":
        on[:] = True
    elif mask == "half":
        on = rng.random(shape) < 0.4
    elif mask == "one":
        on[T // 2, nz - 1, ny - 1, nx - 1] = True
    elif mask == "slab":  # whole tiles stay empty
        on[:, nz // 2:nz // 2 + 3] = rng.random((T, 3, ny, nx)) < 0.5
    f = np.where(on, 0.5 + rng.random(shape), -1.0).astype(np.float32)
    pos = (rng.random((T, 3, 900)) * np.array([nx, ny, nz])[None, :, None]).astype(np.float32)
    a = rng.lognormal(size=(T, A, 900)).astype(np.float32)
    preds = [(0, 0, 0, 0.0, 0.0)]
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x).cuda().contiguous() for x in (f, pos, a)))
        ctx.bin()
        lab, n = ctx.segment(0, T, preds, edges)
        g = ctx.features(0, T, lab, preds, edges)
    finally:
        ctx.close()
    b, olab, on_, o = orc.run_all(f, pos, a, 0, T, preds, edges)
    assert n == on_ == len(g)
    assert np.array_equal(lab.cpu().numpy(), olab)
    for k in ("label", "n_vox", "n_pts"):
        assert np.array_equal(g[k], o[k]), k
    assert np.array_equal(g["sumq"][:, :A], o["sumq"][:, :A])
    np.testing.assert_allclose(g["sum_field"], o["sum_field"], rtol=1e-5)
