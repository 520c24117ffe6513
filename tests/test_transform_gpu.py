"""The per-slice transform (radix-8 passes after a radix-2 or radix-4 one) at every grid size.

The pass structure depends on log2(G / 2) mod 3 and the swizzled buffer on G, so each N_ft from the
smallest to the largest is run through a sum and its gradients against the FP64 oracle.  Bound, relative
to sum|w| max|F| (and its analogue for the gradients): the window's aliasing and fit (3e-7), the
fixed-point grid (2^-31 per source, 1e-8 here), FP32 projections of |u| <= G/2 read by a function of
slope <= D1 (2^-24 D1 / (2 max|F|) of the value, D1 below 60 for these kernels: 2e-6), and the FP32
transform (log2(G) 2^-24: 1e-6): 4e-6 in all.
"""
import numpy as np
import pytest

import oracle
from paper_2410_01316_gb300 import QSPlan
from paper_2410_01316_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 4e-6


@pytest.mark.parametrize("n_ft", [16, 32, 64, 128, 256, 512, 1024, 2048, 4096, 8192])
@pytest.mark.parametrize("proj", ["fp32_fused", "fp32"])
def test_sum_and_gradients_at_every_grid_size(n_ft, proj):
    import torch

    prob = W.tiny(d=3, N=700, M=300, P=9, kernel="gauss", kparam=2.5, n_ft=n_ft, seed=n_ft)
    v = np.random.default_rng(2).standard_normal(prob.M).astype(np.float32)
    x, w, y, vt = (torch.from_numpy(a).cuda() for a in (prob.x, prob.w, prob.y, v))
    with QSPlan(3, "gauss", prob.P, n_ft, prob.R, prob.kparam, dirs=prob.xi, proj=proj, max_n=prob.N,
                max_m=prob.M) as plan:
        s = plan.sum(x, w, y).cpu().numpy().astype(np.float64)
        g = {k: t.cpu().numpy().astype(np.float64) for k, t in plan.grad(x, w, y, vt).items()}
        plan.check()
    t = oracle.tau(prob.kernel, prob.kparam, prob.R)
    c = oracle.coeffs(prob.kernel, prob.kparam, 3, t, n_ft)
    k = np.arange(-n_ft // 2, n_ft // 2)
    D1 = float(np.sum(np.abs(2 * np.pi * k * c)))
    sw, mw = float(np.abs(prob.w).sum()), float(np.abs(prob.w).max())
    sv, mv = float(np.abs(v).sum()), float(np.abs(v).max())
    ref = oracle.o1_grad(prob.x, prob.w, prob.y, v, prob.xi, t, c)
    assert np.max(np.abs(s - oracle.o1_problem(prob))) / sw < TOL
    assert np.max(np.abs(g["w"] - ref["w"])) / sv < TOL
    assert np.max(np.abs(g["y"] - ref["y"])) / (t * sw * mv * D1) < TOL
    assert np.max(np.abs(g["x"] - ref["x"])) / (t * mw * sv * D1) < TOL
