"""The windows of the slice-per-lane kernels are placed by a sample that no regular order of the points defeats.

Two clusters far apart, stored in turn (with periods that divide the distance of evenly spaced samples) and in a random order: the
same sums to within accuracy, and about the same time.  A sample of one cluster only sends half of the points
the slow way, eight atomics on the grid in memory each: 3 to 6 times the time.
"""
import numpy as np
import pytest

from paper_2410_01316_gb300 import QSPlan

pytestmark = pytest.mark.gpu


def _time(f):
    import torch

    best = 1e9
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        f()
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("d,period", [(16, 2), (16, 17), (64, 2)])
def test_points_of_clusters_in_turn(d, period):
    import torch

    N, P = 256 * 782, 512
    gen = torch.Generator(device="cuda").manual_seed(d)
    x, y = (0.3 * torch.randn(N, d, generator=gen, device="cuda") for _ in range(2))
    for a in (x, y):
        a[torch.arange(N, device="cuda") % period != 0] += 8.0 / d**0.5
    order = torch.randperm(N, generator=gen, device="cuda")
    w = torch.full((N,), 1.0 / N, device="cuda")
    R = 1.01 * float(x.norm(dim=1).max() + y.norm(dim=1).max())
    xi = np.random.default_rng(d).standard_normal((P, d))
    xi = (xi / np.linalg.norm(xi, axis=1, keepdims=True)).astype(np.float32)
    with QSPlan(d, "gauss", P, 512, R, 4.0, dirs=xi, max_n=N, max_m=N) as plan:
        assert plan.lanes(N)
        s = plan.sum(x, w, y)
        xs, ys = x[order].contiguous(), y[order].contiguous()
        r = plan.sum(xs, w, ys)
        plan.check()
        assert float((s[order] - r).abs().max()) < 2e-6  # of sum|w| max|F| = 1
        assert _time(lambda: plan.sum(x, w, y)) < 1.5 * _time(lambda: plan.sum(xs, w, ys))
