"""Joins across tile faces against the oracle where tiles are dense: below, at and above the number of
(row, direction) pairs from which a tile's rows are walked direction by direction, and temporal edges
alone, which keep no list."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("edges", [1, 2, 3, 7])
@pytest.mark.parametrize("nx,ny,nz,T,density", [
    (96, 33, 17, 9, 0.3), (96, 33, 17, 9, 0.6), (65, 40, 34, 5, 0.95), (65, 40, 34, 5, 1.0),
    (100, 70, 1, 37, 0.7), (31, 9, 9, 12, 0.9)])
def test_dense_windows(gpu, orc, nx, ny, nz, T, density, edges):
    rng = np.random.default_rng(nx + int(100 * density))
    f = np.where(rng.random((T, nz, ny, nx)) < density, 1.0, -1.0).astype(np.float32)
    pos = (rng.random((T, 3, 700)) * np.array([nx, ny, nz])[None, :, None]).astype(np.float32)
    a = rng.random((T, 1, 700)).astype(np.float32)
    preds = [(0, 0, 0, 0.0, 0.0)]
    o = orc.bin(f.shape, pos, a)
    olab, on = orc.segment(f, o["count"], o["mean"], o["key"], 0, T, preds, edges)
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x).cuda().contiguous() for x in (f, pos, a)))
        ctx.bin()
        lab, n = ctx.segment(0, T, preds, edges)
        assert n == on and np.array_equal(lab.cpu().numpy(), olab)
        labs, ns = ctx.segment_batch([(0, T, preds, edges), (1, T, preds, edges)])
        assert int(ns[0]) == on and np.array_equal(labs[0].cpu().numpy(), olab)
        ctx.set_batch_schedule(gpu.MSF_SCHED_PERSISTENT)
        labs, ns = ctx.segment_batch([(0, T, preds, edges), (1, T, preds, edges)])
        assert int(ns[0]) == on and np.array_equal(labs[0].cpu().numpy(), olab)
    finally:
        ctx.close()
