"""The fixed-point scale of the spread: the same number whichever kernel sums the weights.

Up to 4096 sources every CTA of the spread sums the weights itself, above that a kernel ahead of it does.
Points of weight zero add nothing to any cell, so a problem padded with them to either side of that line has
to give the same bits: signed weights, sums of both kinds of spread (bin moments, N_ft = 256; taps, 2048) and
the gradients, which spread derivative grids.
"""
import numpy as np
import pytest

from paper_2410_01316_gb300 import QSPlan
from paper_2410_01316_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 33, 257, 1000, 1025, 4095])
@pytest.mark.parametrize("n_ft,proj", [(256, "fp32_fused"), (256, "fp32"), (2048, "fp32_fused"), (2048, "fp32")])
def test_sources_of_weight_zero_change_no_bit(N, n_ft, proj):
    import torch

    prob = W.tiny(d=5, N=N, M=301, P=37, kernel="gauss", kparam=2.0, n_ft=n_ft, seed=N)
    prob.w = np.random.default_rng(N).standard_normal(N).astype(np.float32)
    y, v = torch.from_numpy(prob.y).cuda(), torch.randn(prob.M, generator=torch.Generator().manual_seed(1)).cuda()
    results = []
    with QSPlan(5, "gauss", prob.P, n_ft, prob.R, prob.kparam, dirs=prob.xi, proj=proj, max_n=5000, max_m=5000) as plan:
        for n in (N, 4096, 4097, 5000):
            x = np.resize(prob.x, (n, 5))
            w = np.zeros(n, np.float32)
            w[:N] = prob.w
            x, w = torch.from_numpy(x).cuda(), torch.from_numpy(w).cuda()
            s = plan.sum(x, w, y)
            gy = plan.grad(x, w, y, v, want=("y",))["y"]
            plan.check()
            results.append((s, gy))
    for r in results[1:]:
        assert torch.equal(r[0], results[0][0])
        assert torch.equal(r[1], results[0][1])
