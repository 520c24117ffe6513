"""Many equal weights on windows of plain cells: the outermost taps of the window, far below a unit, are not lost.

Nothing cancels in these sums, and with P = 300 slices and over 1e5 sources every random rounding averages out: 2^-22 of
the result's RMS (four roundings to FP32).  Taps that always round to zero are a bias instead, 2.6e-7 to 5.4e-7
here.  The second half of the sources has weight zero and must add nothing.
"""
import numpy as np
import pytest

import oracle
from paper_2410_01316_gb300 import QSPlan
from paper_2410_01316_gb300 import workloads as W
from test_batch_signed_gpu import _sum64

pytestmark = pytest.mark.gpu


def _ball(rng, n):
    x = rng.standard_normal((n, 3))
    return (x / np.linalg.norm(x, axis=1, keepdims=True) * rng.random((n, 1)) ** (1 / 3)).astype(np.float32)


@pytest.mark.parametrize("kernel,n_ft,N,window_kind", [("laplace", 1024, 200003, "es"), ("laplace", 1024, 120001, "kb"),
                                                       ("gauss", 1024, 200003, "es")])
def test_equal_weights(kernel, n_ft, N, window_kind):
    import torch

    rng = np.random.default_rng(N)
    kp = 0.8 if kernel == "gauss" else 1.25
    prob = W.tiny(d=3, N=1000, M=1000, P=300, kernel=kernel, kparam=kp, n_ft=n_ft, seed=3)
    x, y = _ball(rng, N), _ball(rng, 3001)
    R = float(np.linalg.norm(x, axis=1).max() + np.linalg.norm(y, axis=1).max()) * 1.000001
    w = np.full(N, 1.0 / N, np.float32)
    t = oracle.tau(kernel, kp, R)
    ref = _sum64(x, w, y, prob.xi, t, oracle.coeffs(kernel, kp, 3, t, n_ft))
    with QSPlan(3, kernel, 300, n_ft, R, kp, dirs=prob.xi, proj="fp32", max_n=2 * N, max_m=3001, window_kind=window_kind) as plan:
        assert plan.lanes(N)
        for zeros in (0, N):
            xz, wz = np.concatenate([x, x[:zeros]]), np.concatenate([w, np.zeros(zeros, np.float32)])
            s = plan.sum(*(torch.from_numpy(a).cuda() for a in (xz, wz, y))).cpu().numpy()
            plan.check()
            assert np.linalg.norm(s - ref) / np.linalg.norm(ref) < 2.0**-22
