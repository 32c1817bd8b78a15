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
