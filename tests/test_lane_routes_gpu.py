"""Which sums take the slice-per-lane kernels, and that every way through them gives the sum."""
import pytest

from paper_2410_01316_gb300 import QSPlan

pytestmark = pytest.mark.gpu


def _lines(d, P, proj, n_ft=256, kernel="gauss", window=8):
    """The smallest number of points that runs with one slice per lane (None below 2^20 points)."""
    with QSPlan(d, kernel, P, n_ft, 12.0, 0.0 if kernel == "negdist" else 5.0, window=window, dirs="iid", proj=proj,
                max_n=64, max_m=64) as plan:
        lo, hi = 0, 1 << 20
        if not plan.lanes(hi):
            return None
        while hi - lo > 1:
            mid = (lo + hi) // 2
            lo, hi = (lo, mid) if plan.lanes(mid) else (mid, hi)
        return hi


@pytest.mark.parametrize("d,P,proj,pairs", [
    (3, 512, "fp32_fused", 2 << 20), (64, 512, "bf16x3", 2 << 20), (784, 2048, "bf16x3", 2 << 20), (64, 640, "tf32", 2 << 20),
    # fewer than 512 slices: at 2 x 2^20 pairs 0.92 (d = 64) and 0.96 (d = 3) of the point-per-lane kernels' speed
    (3, 320, "fp32_fused", 3 << 20), (64, 320, "bf16x3", 3 << 20), (3, 511, "fp32", 3 << 20),
    (16, 320, "fp32", 3 << 20), (16, 640, "fp32", 3 << 20), (5, 1280, "fp32", 3 << 20), (30, 320, "fp32", 6 << 20),
    (48, 1024, "fp32", 6 << 20)])
def test_lines(d, P, proj, pairs):
    assert _lines(d, P, proj) == -(-pairs // P)


def test_never():
    assert _lines(3, 64, "fp32_fused", window=6) is None      # another window
    assert _lines(100, 512, "fp32") is None                   # FP32 projections beyond d = 64
    assert _lines(3, 512, "fp32_fused", n_ft=2048, kernel="negdist") is None  # windows that would take two walks
    assert _lines(16, 8192, "fp32") == 512                    # never fewer than 512 points
