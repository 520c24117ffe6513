"""The sum over slices of the slice-per-lane interpolation is compensated.

Every slice's value is the same number wherever in its group of lanes the slice lies, so a permutation of
the directions within the groups changes nothing but the order in which the values are added.  With every addition's
error kept (about 2^-47 of the values' sum is lost), the FP32 result can only change where it lies that close to a rounding
boundary: in less than one of a thousand targets, by one unit.  Weights of mean zero make the values some ten
times the result, so that plain FP32 additions change most results.
"""
import numpy as np
import pytest

from paper_2410_01316_gb300 import QSPlan
from paper_2410_01316_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# d = 30: two slices per lane; n_ft = 2048: several windows per slice; 64: tensor-core projections
@pytest.mark.parametrize("d,n_ft,spread_out,proj", [(3, 128, False, "auto"), (16, 256, False, "fp32"), (30, 128, False, "fp32"),
                                                    (32, 1024, True, "fp32_fused"), (32, 2048, True, "fp32"), (64, 512, False, "bf16x3")])
def test_order_of_slices(d, n_ft, spread_out, proj):
    import torch

    P, N, M = 320, 24001, 24007
    prob = W.tiny(d=d, N=N, M=M, P=P, kernel="gauss", kparam=np.sqrt(2.0 * d), n_ft=n_ft, seed=d)
    if spread_out:
        prob.x[:, :2] *= 100.0
        prob.y[:, :2] *= 100.0
        prob.xi[:, 2:] *= 0.02
        prob.xi /= np.linalg.norm(prob.xi, axis=1, keepdims=True)
        prob.R = W.radius(prob.x, prob.y)
        prob.kparam = 50.0
    rng = np.random.default_rng(d)
    w = rng.standard_normal(N)
    w = torch.from_numpy((w - w.mean()).astype(np.float32)).cuda()
    x, y = torch.from_numpy(prob.x).cuda(), torch.from_numpy(prob.y).cuda()
    order = np.concatenate([64 * g + rng.permutation(64) if d == 30 else np.concatenate([64 * g + 32 * h + rng.permutation(32) for h in (0, 1)])
                            for g in range(P // 64)])
    out = []
    for xi in (prob.xi, np.ascontiguousarray(prob.xi[order])):
        with QSPlan(d, "gauss", P, n_ft, prob.R, prob.kparam, dirs=xi, proj=proj, max_n=N, max_m=M) as plan:
            assert plan.lanes(N) and plan.lanes(M)
            out.append(plan.sum(x, w, y).cpu().numpy())
            plan.check()
    differ = out[0] != out[1]
    assert differ.mean() < 1e-3
    assert np.all(np.abs(out[0] - out[1])[differ] <= np.spacing(np.abs(out[0][differ])))
