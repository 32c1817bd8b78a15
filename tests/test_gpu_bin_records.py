"""Binning against the oracle at the edges of the record passes: few buckets (samples sorted per
block) and more than that takes, blocks that end inside a point step, every record width, voxels
with one, two and many records, buckets with more records than a block stages, no sample inside."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,T,P,A,crowd", [
    (32, 32, 32, 3, 4096, 1, 0.0), (33, 31, 7, 4, 4097, 2, 0.3), (64, 64, 8, 2, 20000, 0, 0.2),
    (61, 17, 9, 3, 2049, 3, 0.5), (40, 40, 40, 2, 30000, 4, 0.1), (24, 24, 24, 2, 9000, 6, 0.4),
    (24, 24, 24, 2, 9000, 7, 0.4), (30, 20, 10, 2, 6000, 8, 0.9), (16, 16, 16, 2, 50000, 2, 0.0),
    (161, 161, 161, 2, 9000, 2, 0.1), (163, 162, 161, 2, 9000, 2, 0.1),
    (129, 128, 128, 1, 5000, 4, 0.2), (10, 10, 10, 2, 700, 2, -1.0)])
def test_bins_match_oracle(gpu, orc, nx, ny, nz, T, P, A, crowd):
    rng = np.random.default_rng(nx + P + A)
    f = np.zeros((T, nz, ny, nx), np.float32)
    box = np.array([nx, ny, nz])[None, :, None]
    pos = (rng.random((T, 3, P)) * (1.01 * box)).astype(np.float32)
    if crowd < 0:
        pos -= 2.0 * np.array([nx, ny, nz], np.float32)[None, :, None]  # all outside
    else:  # some samples share a few voxels
        m = rng.random((T, P)) < crowd
        spot = np.floor(rng.random((T, 3, 5)) * box) + 0.25
        pick = rng.integers(0, 5, size=(T, P))
        for t in range(T):
            pos[t][:, m[t]] = spot[t][:, pick[t]][:, m[t]]
    a = (rng.normal(size=(T, A, P)) * 10.0 ** rng.integers(-6, 3, size=(T, A, P))).astype(np.float32)
    if A:
        a.reshape(-1)[::997] = np.nan
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x).cuda().contiguous() for x in (f, pos, a)))
        st = ctx.bin(keep_sumq=True)
        key, count, mean, sumq = ctx.bins("cpu", sumq=True)
    finally:
        ctx.close()
    o = orc.bin(f.shape, pos, a, keep_sumq=True)
    assert np.array_equal(key.numpy(), o["key"])
    assert st.in_domain == int((o["key"] >= 0).sum())
    assert np.array_equal(count.numpy(), o["count"])
    if A:
        assert np.array_equal(sumq.numpy(), o["sumq"])
        assert np.array_equal(mean.numpy().view(np.uint32), np.asarray(o["mean"]).view(np.uint32)) \
            or np.array_equal(mean.numpy(), o["mean"], equal_nan=True)
