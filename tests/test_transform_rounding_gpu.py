"""Rounding of the per-slice transform, seen in sums whose terms do not cancel.

With equal weights and a positive kernel the result is as large as its terms, and P slices average the
rounding of each. What is left over then comes from the few roundings of every stage: at most twice the RMS rounding
to FP32 of the result itself, 2 x 2^-24 / sqrt(3) = 6.9e-8 of its RMS.  Twiddle factors formed by a product of two
table entries instead of read from the table take the transform over that.
"""
import math

import numpy as np
import pytest

import oracle
from paper_2410_01316_gb300 import QSPlan
from paper_2410_01316_gb300 import workloads as W
from test_batch_signed_gpu import _sum64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ft", [128, 256, 512])
def test_equal_weights(n_ft):
    import torch

    rel = []
    for seed in range(4):
        rng = np.random.default_rng(seed)
        prob = W.tiny(d=5, N=3000, M=2000, P=100, kernel="gauss", kparam=math.sqrt(10.0), n_ft=n_ft, seed=seed)
        prob.x, prob.y = (rng.standard_normal((n, 5)).astype(np.float32) for n in (3000, 2000))
        prob.R = W.radius(prob.x, prob.y)
        prob.w = np.full(3000, 1.0 / 3000, np.float32)
        x, w, y = (torch.from_numpy(a).cuda() for a in (prob.x, prob.w, prob.y))
        with QSPlan(5, "gauss", 100, n_ft, prob.R, prob.kparam, dirs=prob.xi, max_n=3000, max_m=2000) as plan:
            s = plan.sum(x, w, y).cpu().numpy().astype(np.float64)
            plan.check()
        t = oracle.tau("gauss", prob.kparam, prob.R)
        ref = _sum64(prob.x, prob.w, prob.y, prob.xi, t, oracle.coeffs("gauss", prob.kparam, 5, t, n_ft))
        rel.append(np.linalg.norm(s - ref) / np.linalg.norm(ref))
    assert np.mean(rel) < 2 * 2.0**-24 / math.sqrt(3.0), rel
