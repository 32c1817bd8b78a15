"""Binning and queries where device memory is short: the records' second copy of the voxel pairs is left
out where it does not fit, or given back to a later call, and the results stay the same. Memory is
taken with plain allocations, all of it freed again."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture
def fill():
    """fill(leave): allocations that leave about `leave` bytes of the device free (20 MB is the
    allocator's step); fill(None) frees them, as the end of the test does."""
    held = []

    def f(leave):
        held.clear()
        torch.cuda.empty_cache()
        for size in (16 << 30, 1 << 30, 100 * MB, 20 * MB) if leave is not None else ():
            while torch.cuda.mem_get_info()[0] > leave + size + 8 * MB:
                held.append(torch.empty(size, dtype=torch.uint8, device="cuda"))

    yield f
    f(None)


def _data(A, P=2 << 20, T=8, n=64):
    g = torch.Generator(device="cuda")
    g.manual_seed(A)
    field = torch.randn((T, n, n, n), generator=g, device="cuda")
    pos = torch.rand((T, 3, P), generator=g, device="cuda") * n
    return field, pos, torch.rand((T, A, P), generator=g, device="cuda")


def _answers(ctx, crit_args, labels, gpu):
    n = gpu.msf_segment(ctx.h, gpu.make_criteria(*crit_args), labels)
    f = ctx.features(crit_args[0], crit_args[1], labels, *crit_args[2:])
    return n, labels.cpu().numpy().copy(), f


def _same(a, b, A):
    assert a[0] == b[0] and np.array_equal(a[1], b[1])
    for k in ("label", "n_vox", "n_pts", "sumq", "bbox_min", "bbox_max", "mean_attr"):
        assert np.array_equal(a[2][k], b[2][k], equal_nan=k == "mean_attr"), k
    np.testing.assert_allclose(a[2]["std_attr"][:, :A], b[2]["std_attr"][:, :A], rtol=1e-6,
                               atol=1e-7, equal_nan=True)


@pytest.mark.parametrize("A", [1, 4, 8])
def test_pairs_left_out_or_given_back(gpu, fill, A):
    field, pos, attr = _data(A)
    T, n = field.shape[0], field.shape[1]
    args = (0, T, [(0, 0, 0, 1.2, 0.0)], 7)
    labels = torch.empty(field.shape, dtype=torch.int32, device="cuda")
    queries = [(t & 1, T, [(0, 0, 0, 1.0 + 0.05 * t, 0.0)], 7) for t in range(16)]
    out = [torch.empty((T - (t & 1), n, n, n), dtype=torch.int32, device="cuda") for t in range(16)]
    other = gpu.Context(0)               # (also loads every kernel's code while there is room)
    try:
        other.load(field, pos, attr)
        other.bin()
        other.segment_batch(queries, out)
        want_batch = [x.cpu() for x in out]
    finally:
        other.close()
    first = gpu.Context(0)
    try:
        first.load(field, pos, attr)
        first.bin()
        want = _answers(first, args, labels, gpu)
        # given back: a batch's scratch (about 110 MB) takes the pairs' place (134 MB)
        torch.cuda.synchronize()
        fill(32 * MB)
        assert torch.cuda.mem_get_info()[0] < 64 * MB
        first.segment_batch(queries, out)
        fill(None)
        for x, y in zip(out, want_batch):
            assert torch.equal(x.cpu(), y)
        _same(_answers(first, args, labels, gpu), want, A)
    finally:
        first.close()
    # left out: a new context, with room for everything but the pairs
    NR = pos.shape[0] * pos.shape[2]
    rec = 16 if A <= 2 else 32 if A <= 6 else 48
    need = NR * (12 + 4 * A + 4 + rec) + field.numel() * (8 + 4 * A) + 64 * MB
    fill(need + NR * 8 // 2)
    ctx = gpu.Context(0)
    try:
        ctx.load(field, pos, attr)
        ctx.bin()
        _same(_answers(ctx, args, labels, gpu), want, A)
        fill(None)
        ctx.bin()                         # with room again
        _same(_answers(ctx, args, labels, gpu), want, A)
    finally:
        ctx.close()
