"""Per-cluster summaries of long rows, which several blocks share, and of row lengths around a block's
columns."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,T", [(300001, 1, 1, 3), (70000, 2, 1, 2), (1023, 3, 2, 2),
                                        (1024, 3, 2, 2), (1025, 3, 2, 2), (255, 1, 1, 1),
                                        (257, 40, 1, 9), (5000, 40, 1, 4), (1, 1, 40000, 3)])
@pytest.mark.parametrize("labels", ["random", "along"])
def test_long_rows_match_oracle(gpu, orc, nx, ny, nz, T, labels):
    rng = np.random.default_rng(nx + T)
    K = 300
    f = rng.normal(1.0, 2.0, size=(T, nz, ny, nx)).astype(np.float32)
    f.reshape(-1)[::997] = np.nan
    fl = rng.integers(-1, K, size=f.shape).astype(np.int32)
    if labels == "along":
        fl = (np.arange(f.size, dtype=np.int64) * K // f.size).astype(np.int32).reshape(f.shape)
    pos = (rng.random((T, 3, 50)) * np.array([nx, ny, nz])[None, :, None]).astype(np.float32)
    a = rng.lognormal(size=(T, 1, 50)).astype(np.float32)
    ctx = gpu.Context(0)
    try:
        ctx.load(*(torch.as_tensor(x).cuda().contiguous() for x in (f, pos, a)))
        ctx.bin()
        g = ctx.cluster_stats(0, T, 0, torch.as_tensor(fl).cuda(), None, K)
        key = ctx.bins("cpu")[0].numpy()
    finally:
        ctx.close()
    o = orc.cluster_stats(f, pos, a, key, 0, T, 0, fl, None, K)
    for k in ("n_field", "n_point", "lo", "hi"):
        assert np.array_equal(g[k], o[k]), k
    assert np.array_equal(g["mean_field"], o["mean_field"], equal_nan=True)
    np.testing.assert_allclose(g["std_field"], o["std_field"], rtol=1e-9, atol=1e-12, equal_nan=True)


def test_few_long_rows_fill_the_gpu(gpu):
    """Eight rows of 2^20 values take no longer than the same values in rows of 1024 by more than a
    factor of four (with a block per row they took forty times as long)."""
    import time
    times = []
    for nx, ny in ((1 << 20, 1), (1 << 10, 1 << 10)):
        f = torch.rand((8, 1, ny, nx), device="cuda")
        fl = torch.randint(0, 1000, f.shape, dtype=torch.int32, device="cuda")
        ctx = gpu.Context(0)
        try:
            ctx.load(f, torch.full((8, 3, 1), 0.5, device="cuda"), torch.ones((8, 1, 1), device="cuda"))
            ctx.bin()
            best = 1e9
            for _ in range(6):
                torch.cuda.synchronize()
                t = time.perf_counter()
                ctx.cluster_stats(0, 8, 0, fl, None, 1000)
                best = min(best, time.perf_counter() - t)
        finally:
            ctx.close()
        times.append(best)
    assert times[0] < 4 * times[1], times
