"""Feature statistics against the oracle where the grouping has edges: tiles filled by one feature,
tiles of single-voxel features (more than the group table takes), features around a thread's and a
warp's share, labels on both sides of the one-launch ranking's limit, many attributes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,T,A,P,edges,mask", [
    (32, 32, 16, 5, 1, 3000, 7, "all"), (40, 17, 9, 6, 2, 3000, 0, "all"),
    (64, 16, 16, 4, 1, 2000, 1, "checker"), (33, 31, 7, 9, 3, 4000, 3, "sparse"),
    (96, 33, 1, 40, 2, 3000, 3, "half"), (33, 20, 11, 3, 8, 2500, 7, "half"),
    (33, 20, 11, 3, 5, 2500, 3, "blocks"), (128, 96, 64, 2, 1, 20000, 3, "sparse"),
    (160, 128, 80, 1, 0, 5000, 1, "sparse")])
def test_features_match_oracle(gpu, orc, nx, ny, nz, T, A, P, edges, mask):
    rng = np.random.default_rng(nx + 7 * T + A)
    f = rng.normal(3.0, 1.0, size=(T, nz, ny, nx)).astype(np.float32)
    i = np.indices(f.shape)
    on = {"all": np.ones(f.shape, bool), "checker": (i[1] + i[2] + i[3]) % 2 == 0,
          "sparse": rng.random(f.shape) < 0.02, "half": rng.random(f.shape) < 0.4,
          "blocks": ((i[3] // 3 + i[2] // 4 + i[1]) % 2 == 0) & (i[3] % 7 > 0)}[mask]
    f = np.where(on, np.abs(f) + 0.5, -1.0).astype(np.float32)
    pos = (rng.random((T, 3, P)) * np.array([nx, ny, nz])[None, :, None]).astype(np.float32)
    a = rng.lognormal(size=(T, A, P)).astype(np.float32)
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
    assert np.array_equal(np.concatenate([g["bbox_min"], g["bbox_max"]], 1), o["bbox"])
    assert np.array_equal(g["sumq"][:, :A], o["sumq"][:, :A])
    for k in ("sum_field", "mean_field", "min_field", "max_field", "centroid"):
        np.testing.assert_allclose(g[k], o[k], rtol=1e-5, err_msg=k)
    # a deviation carries the rounding of the mean's square (fp64): about 1e-8 of the magnitude
    np.testing.assert_allclose(g["std_field"], o["std_field"], rtol=1e-5, atol=1e-6)
    np.testing.assert_allclose(g["mean_attr"][:, :A], o["mean_attr"][:, :A], rtol=1e-5)
    np.testing.assert_allclose(g["std_attr"][:, :A], o["std_attr"][:, :A], rtol=1e-5, atol=1e-6)
