"""The largest problems that qs_sum_noalloc takes: grids, tables and partial sums of exactly 16 MiB.

The layout up to the partial sums (flag and scale 512 B, window transform, coefficients, filter, twiddles, directions and
grids, each rounded up to 256 B) and two partial sums per target fill 16 MiB to the byte; W = 6, whose kernels have
one point per lane whatever the size.
"""
import ctypes

import numpy as np
import pytest

from paper_2410_01316_gb300 import QSPlan, _lib
from paper_2410_01316_gb300 import workloads as W
from test_zz_no_alloc import _desc, _norm

pytestmark = pytest.mark.gpu


def test_sixteen_mebibytes_still_fit():
    import torch

    n_ft, P, d = 512, 8, 3
    up = lambda b: (b + 255) // 256 * 256
    fixed = 512 + up((n_ft // 2 + 1) * 8) + up(n_ft * 8) + up((n_ft + 1) * 4) + up(n_ft * 8) + up(P * d * 4) + up(P * 2 * n_ft * 4)
    M = ((16 << 20) - fixed) // 8
    prob = W.tiny(d=d, N=1000, M=1000, P=P, kernel="gauss", kparam=1.0, n_ft=n_ft, seed=2)
    prob.window = 6
    x, w = torch.from_numpy(prob.x).cuda(), torch.from_numpy(prob.w).cuda()
    y = torch.from_numpy(np.resize(prob.y, (M + 1, d))).cuda()
    lib, desc, out = _lib.load(), _desc(prob), torch.full((M,), float("nan"), device="cuda")
    dirs = torch.from_numpy(prob.xi).cuda()
    call = lambda m, o: lib.qs_sum_noalloc(ctypes.byref(desc), dirs.data_ptr(), x.data_ptr(), 1000, w.data_ptr(), y.data_ptr(), m,
                                           o.data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert call(M, out) == 0, lib.qs_last_error().decode()
    with QSPlan(d, "gauss", P, n_ft, prob.R, prob.kparam, dirs=prob.xi, window=6, proj="fp32_fused", max_n=1000, max_m=M) as plan:
        ref = plan.sum(x, w, y[:M])
        plan.check()
    assert float((out - ref).abs().max()) / _norm(prob, True) < 1e-6
    assert call(M + 1, torch.empty(M + 1, device="cuda")) == 6
