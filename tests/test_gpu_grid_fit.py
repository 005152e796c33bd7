"""The grid fit against the plain iteration in the same arithmetic (fp32 distances in coordinate order, lowest index on
ties, fp64 means): skipped scans, moved samples and the split over blocks and warps must not show."""
import numpy as np
import pytest
import torch

import paper_2411_17525_b200 as hb
from tests import gpu_util as U

pytestmark = pytest.mark.gpu


def plain_lloyd(p, n, x, max_iters, cells=None):
    c = x[:n].copy()
    old = np.full(len(x), -1)
    for it in range(1, max_iters + 1):
        a = np.empty(len(x), dtype=np.int64)
        err = 0.0
        for i in range(0, len(x), 4096):
            e = (x[i:i + 4096, None, :] - c[None]).astype(np.float64)          # fp32 differences, widened
            d = (e[..., 0] ** 2).astype(np.float32)
            for k in range(1, p):
                d = (e[..., k] ** 2 + d).astype(np.float32)                    # one rounding, as a fused multiply-add
            d = np.where(np.isnan(d), np.float32(np.inf), d)                       # (never below infinity: index 0 when all are)
            a[i:i + 4096] = d.argmin(1)
            err += float(d.min(1).astype(np.float64).sum())
        if np.array_equal(a, old):
            return c, err, it
        old = a
        size = np.bincount(a, minlength=n)
        if cells is not None:                                                      # sizes and sums of magnitudes behind the centres
            cells[0][:] = size
        for k in range(p):
            if cells is not None:
                cells[1][:, k] = np.bincount(a, weights=np.abs(x[:, k].astype(np.float64)), minlength=n)
            s = np.bincount(a, weights=x[:, k].astype(np.float64), minlength=n)
            c[size > 0, k] = (s[size > 0] / size[size > 0]).astype(np.float32)
    return c, err, -max_iters


@pytest.mark.parametrize("p,n,m,max_iters", [
    (1, 1, 1, 5), (1, 4, 31, 50), (2, 16, 33, 50),          # a part of a warp, one sample more than a warp
    (2, 256, 257, 50),                                      # cells of one sample
    (2, 65, 151559, 40), (1, 80, 40000, 60), (2, 300, 30000, 80), (3, 512, 20000, 30),                                   # more than one sample per lane on some warps
    (1, 16, 8192, 400), (3, 830, 4000, 60), (4, 33, 20000, 60), (4, 4096, 5000, 4),
])
def test_fit_follows_the_plain_iteration(p, n, m, max_iters):
    x = np.random.default_rng(7 * n + m).standard_normal((m, p)).astype(np.float32)
    x[m // 2:m // 2 + 2] = x[0]                             # (equal samples: equal centres when both are among the first n)
    c, err, iters = plain_lloyd(p, n, x, max_iters)
    t = torch.from_numpy(x).to(U.dev())
    grid, mse, it = hb.higgs_make_grid(p, n, t, max_iters=max_iters)
    again, _, _ = hb.higgs_make_grid(p, n, t, max_iters=max_iters)
    assert hb.higgs_device_status() == hb.HIGGS_OK
    assert int(it) == iters
    want = c[np.lexsort(c.T[::-1])]
    assert np.max(np.abs(grid.cpu().numpy() - want)) <= 2.0 ** -22              # an fp32 rounding of a mean of size <= 4
    assert abs(float(mse) - err / (m * p)) <= 1e-6 * err / (m * p) + 1e-30
    assert torch.equal(grid, again)


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf"), 1e30])
@pytest.mark.parametrize("p,n,m", [(1, 16, 300), (2, 256, 4133), (2, 600, 5000), (4, 40, 333)])
def test_samples_without_a_nearest_centre(p, n, m, bad):
    """A sample whose distances are all NaN or infinite belongs to cell 0, whichever way it is scanned."""
    x = np.random.default_rng(n).standard_normal((m, p)).astype(np.float32)
    x[n + 3, p - 1] = x[m - 1, 0] = bad
    grid, mse, it = hb.higgs_make_grid(p, n, torch.from_numpy(x).to(U.dev()), max_iters=12)
    assert hb.higgs_device_status() == hb.HIGGS_OK
    assert 1 <= abs(int(it)) <= 12
    with np.errstate(all="ignore"):
        c, err, iters = plain_lloyd(p, n, x, 12)
    assert int(it) == iters
    assert np.isinf(float(mse)) if np.isinf(err) else abs(float(mse) - err / (m * p)) <= 1e-6 * err / (m * p)
    if not np.isnan(bad):                                   # (a NaN has no place in the order of the centres)
        want = c[np.lexsort(c.T[::-1])]
        assert np.allclose(grid.cpu().numpy(), want, rtol=2.0 ** -22, atol=2.0 ** -22)


@pytest.mark.parametrize("p,n,m,case", [(1, 16, 4000, "outlier"), (2, 256, 70000, "outlier"), (2, 256, 33, "few"), (2, 600, 5000, "spread"),
                                        (4, 100, 9000, "spread"), (1, 64, 3000, "tiny"), (3, 300, 4000, "huge")])
def test_samples_of_another_range(p, n, m, case):
    """Sets that 64-bit fixed-point sums would round: their means are those of fp64 sums."""
    if case == "few":
        n = 16
    rng = np.random.default_rng(n)
    x = rng.standard_normal((m, p))
    if case == "spread":
        x *= 10.0 ** rng.uniform(-12, 12, (m, 1))
    x = (x * {"tiny": 1e-25, "huge": 1e18}.get(case, 1.0)).astype(np.float32)
    if case in ("outlier", "few"):
        x[m - 2, 0], x[n + 2, p - 1] = 3e15, -1e15
    size, mag = np.zeros(n), np.zeros((n, p))
    c, err, iters = plain_lloyd(p, n, x, 40, cells=(size, mag))
    grid, mse, it = hb.higgs_make_grid(p, n, torch.from_numpy(x).to(U.dev()), max_iters=40)
    assert hb.higgs_device_status() == hb.HIGGS_OK
    assert int(it) == iters
    # per cell: fp64 sums of its samples in another order, the sum of magnitudes over the size, then one rounding to fp32
    bound = size[:, None] * 2.0 ** -53 * mag / np.maximum(size, 1)[:, None] + 2.0 ** -23 * np.abs(c)
    order = np.lexsort(c.T[::-1])
    assert np.all(np.abs(grid.cpu().numpy().astype(np.float64) - c[order]) <= bound[order])
    assert abs(float(mse) - err / (m * p)) <= 1e-6 * err / (m * p) + 1e-30


@pytest.mark.parametrize("p,n,m", [(1, 4, 31), (2, 256, 30000), (2, 600, 5000)])
@pytest.mark.parametrize("value", [0.5, float("inf")])
def test_a_barrier_that_runs_out(p, n, m, value):
    """Blocks that wait for one arrival too many give up: a reported timeout and defined outputs, and the next fit is none the worse."""
    x = np.random.default_rng(m).standard_normal((m, p)).astype(np.float32)
    x[m - 1, 0] = value                                     # (infinite: the kernel for sample sets of any range)
    t = torch.from_numpy(x).to(U.dev())
    grid, mse, it = hb.higgs_selftest_grid_fit(0, p, n, t)
    assert hb.higgs_device_status() == hb.HIGGS_ERR_TIMEOUT
    assert int(it) < 0 and np.isnan(float(mse))
    assert np.array_equal(grid.cpu().numpy(), x[:n][np.lexsort(x[:n].T[::-1])])
    _, mse, it = hb.higgs_make_grid(p, n, t, max_iters=20)
    assert hb.higgs_device_status() == hb.HIGGS_OK
    assert int(it) != 0 and not np.isnan(float(mse))


@pytest.mark.parametrize("p,n,m", [(1, 16, 8192), (2, 256, 70000)])
@pytest.mark.parametrize("value", [0.5, 1e15])
def test_fewer_resident_blocks_than_asked_for(p, n, m, value):
    """A launch that the runtime refuses because not all its blocks are resident is repeated with fewer: same result."""
    x = np.random.default_rng(m).standard_normal((m, p)).astype(np.float32)
    x[m - 1, 0] = value
    t = torch.from_numpy(x).to(U.dev())
    got, want = hb.higgs_selftest_grid_fit(1, p, n, t), hb.higgs_make_grid(p, n, t, max_iters=100)
    assert hb.higgs_device_status() == hb.HIGGS_OK
    assert int(got[2]) == int(want[2])
    if value < 1:
        assert torch.equal(got[0], want[0])
    else:                                                   # (fp64 sums in any order, one rounding to fp32)
        assert torch.allclose(got[0], want[0], rtol=2.0 ** -22, atol=2.0 ** -22)


@pytest.mark.parametrize("p,n,m", [(1, 4, 31), (2, 16, 8192), (1, 64, 3000), (2, 65, 9000), (1, 256, 4000), (2, 512, 5001), (2, 600, 5000)])
def test_the_variant_for_large_sets(p, n, m):
    """Plain iterations in turn with bounded ones, where bounds pay and where they do not."""
    x = np.random.default_rng(3 * n + m).standard_normal((m, p)).astype(np.float32)
    c, err, iters = plain_lloyd(p, n, x, 100)
    grid, mse, it = hb.higgs_selftest_grid_fit(2, p, n, torch.from_numpy(x).to(U.dev()))
    assert hb.higgs_device_status() == hb.HIGGS_OK
    assert int(it) == iters
    assert np.max(np.abs(grid.cpu().numpy() - c[np.lexsort(c.T[::-1])])) <= 2.0 ** -22
    assert abs(float(mse) - err / (m * p)) <= 1e-6 * err / (m * p) + 1e-30
