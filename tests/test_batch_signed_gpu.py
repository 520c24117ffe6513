"""Concurrent batches of uneven problems with signed weights, against 64 bits and relative to the result.

The problems are those that a batch is made of: d = 3, 16, 64, few slices, up to 40000 points, weights N(0, 1)
as they are and with mean zero, where the result cancels to a few percent of ||w||.  All targets are compared.

Bound on the RMS error.  The spread rounds N W contributions to units of sum|w| 2^-30 (variance 1/12 each, at
both ends of a mirrored pair, so a factor 2), and P slices average: 2 sum|w| 2^-30 sqrt(8 N / 12 / P).  What is rounded relative to a
contribution (projections, taps, transform) is independent from source to source: 2^-16 of ||w|| for the
BF16x3 projections of d = 64, over sqrt(P) slices; 2^-20 of ||w|| / sqrt(P) for FP32.
"""
import math

import numpy as np
import pytest

import oracle
from paper_2410_01316_gb300 import QSBatch, QSPlan
from paper_2410_01316_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SPECS = [(d, N, M, P, n_ft) for i, (d, P) in enumerate([(3, 128), (16, 128), (64, 128), (3, 256), (16, 256), (64, 256)])
         for N, M, n_ft in [(40000, 301, 256), (33001, 20011, 1024), (3001, 12007, 512), (700 + i, 35000, 512)]]


def _sum64(x, w, y, xi, t, c):
    """(1/P) sum_p sum_k c_k e^(2 pi i k t b) sum_n w_n e^(-2 pi i k t a), in 64 bits on the GPU."""
    import torch

    k = np.arange(-len(c) // 2, len(c) // 2)
    keep = np.abs(c) > 1e-14 * np.abs(c).sum()  # the others add less than 1e-11 of the sum
    kk = torch.from_numpy(k[keep].astype(np.float64)).cuda()
    ck = torch.from_numpy(np.ascontiguousarray(c[keep], dtype=np.float64)).cuda()
    X, Y, ww, D = (torch.from_numpy(np.ascontiguousarray(a)).double().cuda() for a in (x, y, w, xi))
    s = torch.zeros(len(y), dtype=torch.float64, device="cuda")
    for p in range(len(xi)):
        a, b = 2 * math.pi * t * (X @ D[p]), 2 * math.pi * t * (Y @ D[p])
        h = torch.zeros(len(kk), dtype=torch.complex128, device="cuda")
        for q in range(0, len(a), 16384):
            ph = kk[:, None] * a[None, q:q + 16384]
            h += torch.complex((torch.cos(ph) @ ww[q:q + 16384]), -(torch.sin(ph) @ ww[q:q + 16384]))
        h *= ck
        for q in range(0, len(b), 16384):
            ph = b[q:q + 16384, None] * kk[None, :]
            s[q:q + 16384] += torch.cos(ph) @ h.real - torch.sin(ph) @ h.imag
    return s.cpu().numpy() / len(xi)


@pytest.mark.parametrize("mean_zero", [False, True])
def test_signed_uneven_batch(mean_zero):
    import torch

    probs, plans, data = [], [], []
    for i, (d, N, M, P, n_ft) in enumerate(SPECS):
        prob = W.tiny(d=d, N=N, M=M, P=P, kernel="gauss", kparam=math.sqrt(2 * d), n_ft=n_ft, seed=40 + i)
        rng = np.random.default_rng(i)
        prob.x, prob.y = (rng.standard_normal((n, d)).astype(np.float32) for n in (N, M))
        prob.R = W.radius(prob.x, prob.y)
        prob.w = rng.standard_normal(N).astype(np.float32)
        if mean_zero:
            prob.w -= prob.w.mean(dtype=np.float64).astype(np.float32)
        plan = QSPlan(d, "gauss", P, n_ft, prob.R, prob.kparam, dirs=prob.xi, max_n=N, max_m=M)
        assert not plan.lanes(N) and not plan.lanes(M)
        probs.append(prob)
        plans.append(plan)
        data.append((*(torch.from_numpy(a).cuda() for a in (prob.x, prob.w, prob.y)), torch.empty(M, device="cuda")))
    own = [plan.sum(x, w, y) for plan, (x, w, y, _) in zip(plans, data)]
    batch = QSBatch(plans)
    batch.set_mode(concurrent=True)
    batch.sum(data)
    batch.check()
    for prob, (d, N, M, P, n_ft), o, (_, _, _, out) in zip(probs, SPECS, own, data):
        assert torch.equal(o, out)
        t = oracle.tau(prob.kernel, prob.kparam, prob.R)
        ref = _sum64(prob.x, prob.w, prob.y, prob.xi, t, oracle.coeffs(prob.kernel, prob.kparam, d, t, n_ft))
        w = prob.w.astype(np.float64)
        err = np.sqrt(np.mean((out.cpu().numpy() - ref) ** 2))
        bound = (2 * np.abs(w).sum() * 2.0**-30 * math.sqrt(8 * N / 12 / P)
                 + np.linalg.norm(w) * (2.0**-16 if d == 64 else 2.0**-20) / math.sqrt(P))
        rms = np.sqrt(np.mean(ref**2))
        print(f"d={d} N={N} M={M} P={P}: error {err / rms:.1e} of the result, {err / bound:.2f} of the bound")
        assert err < bound, (d, N, M, P, n_ft)
    batch.close()
    for plan in plans:
        plan.close()


def test_few_slices_keep_the_point_per_lane_kernels():
    # up to 256 slices the line is at 48 x 1024 points, above that at the products of points and slices
    with QSPlan(16, "gauss", 256, 512, 12.0, 5.0, max_n=1 << 20, max_m=1 << 20) as plan:
        assert [plan.lanes(n) for n in (0, 12288, 40000, 49151, 49152, 200000)] == [False] * 4 + [True] * 2
    with QSPlan(16, "gauss", 257, 512, 12.0, 5.0, max_n=1 << 20, max_m=1 << 20) as plan:
        assert [plan.lanes(n) for n in (1000, 40000)] == [False, True]
