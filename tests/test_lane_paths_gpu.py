"""Every way through the slice-per-lane kernels, at sizes where they are sure to run.

Sums of signed weights with mean zero, so that the result is a few percent of ||w||, every target against 64 bits.  Bound on the
RMS error: what is rounded relative to a contribution is independent from source to source, eps ||w|| / sqrt(P), with
eps = 2^-20 for FP32 projections, 2^-16 for BF16x3 and 2^-8 for TF32 (|u| 2^-11 cells, the values' slope of 0.1 per cell);
a cell is rounded to units of sum|w| 2^-30 once per CTA that adds a window to it (at most 152 per group, and 4 times as many where
windows of plain cells take 16384 points each), G cells, P slices.  Sources or targets with one point per lane round all 8 taps
of all N sources instead.
"""
import ctypes
import math

import numpy as np
import pytest

import oracle
from paper_2410_01316_gb300 import QSPlan, _lib
from paper_2410_01316_gb300 import workloads as W
from test_batch_signed_gpu import _sum64
from test_lane_gpu import _check
from test_zz_no_alloc import _desc

pytestmark = pytest.mark.gpu

EPS = {"fp32": 2.0**-20, "fp32_fused": 2.0**-20, "bf16x3": 2.0**-16, "tf32": 2.0**-8}


def _problem(d, N, M, P, n_ft, seed, kernel="gauss"):
    prob = W.tiny(d=d, N=N, M=M, P=P, kernel=kernel, kparam=math.sqrt(2 * d), n_ft=n_ft, seed=seed)
    rng = np.random.default_rng(seed)
    prob.x, prob.y = (rng.standard_normal((n, d)).astype(np.float32) for n in (N, M))
    prob.R = W.radius(prob.x, prob.y)
    w = rng.standard_normal(N)
    prob.w = (w - w.mean()).astype(np.float32)
    return prob


def _bound(prob, proj, lane_sources):
    w = prob.w.astype(np.float64)
    roundings = 608 * 2 * prob.n_ft if lane_sources else 8 * prob.N
    return (EPS[proj] * np.linalg.norm(w) + 2 * np.abs(w).sum() * 2.0**-30 * math.sqrt(roundings / 12)) / math.sqrt(prob.P)


def _reference(prob):
    t = oracle.tau(prob.kernel, prob.kparam, prob.R)
    return _sum64(prob.x, prob.w, prob.y, prob.xi, t, oracle.coeffs(prob.kernel, prob.kparam, prob.d, t, prob.n_ft))


@pytest.mark.parametrize("d,proj", [(3, "fp32_fused"), (7, "fp32"), (16, "fp32"), (30, "fp32"), (30, "fp32_fused"), (64, "fp32"),
                                    (64, "bf16x3"), (100, "bf16x3"), (48, "tf32")])
@pytest.mark.parametrize("N,M", [(26003, 25001), (26003, 700), (700, 26003)])
def test_both_kinds_and_each_of_them(d, proj, N, M):
    import torch

    P = 290
    prob = _problem(d, N, M, P, 256, d + N)
    x, w, y = (torch.from_numpy(a).cuda() for a in (prob.x, prob.w, prob.y))
    with QSPlan(d, "gauss", P, 256, prob.R, prob.kparam, dirs=prob.xi, proj=proj, max_n=N, max_m=M) as plan:
        assert plan.lanes(N) == (N > 10000) and plan.lanes(M) == (M > 10000)
        s = plan.sum(x, w, y)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            g = plan.sum(x, w, y)
        graph.replay()
        assert torch.equal(g, s)
        plan.check()
        assert np.array_equal(plan.sum_host(prob.x, prob.w, prob.y), s.cpu().numpy())
    err = np.sqrt(np.mean((s.cpu().numpy() - _reference(prob)) ** 2))
    assert err < _bound(prob, proj, N > 10000)


@pytest.mark.parametrize("n_ft,window_kind", [(128, "kb"), (512, "kb"), (1024, "es"), (2048, "es")])
@pytest.mark.parametrize("d,proj", [(16, "fp32"), (64, "bf16x3")])
def test_windows_and_grids(n_ft, window_kind, d, proj):
    import torch

    prob = _problem(d, 24001, 24011, 300, n_ft, n_ft)
    with QSPlan(d, "gauss", 300, n_ft, prob.R, prob.kparam, dirs=prob.xi, proj=proj, max_n=prob.N, max_m=prob.M,
                window_kind=window_kind) as plan:
        assert plan.lanes(prob.N) and plan.lanes(prob.M)
        s = plan.sum(*(torch.from_numpy(a).cuda() for a in (prob.x, prob.w, prob.y))).cpu().numpy()
        plan.check()
    assert np.sqrt(np.mean((s - _reference(prob)) ** 2)) < _bound(prob, proj, True)


# gradients, sums and repeated calls as in test_lane_gpu.py, at 320 slices
@pytest.mark.parametrize("d,N,M,proj,shift", [(1, 9999, 10111, "fp32_fused", 0), (4, 11003, 10007, "fp32", 1), (6, 12001, 300, "fp32", 1),
                                              (16, 300, 11999, "fp32", 0), (30, 21001, 20999, "fp32", 1), (48, 20003, 400, "fp32", 0),
                                              (64, 20005, 20001, "fp32", 0), (64, 10007, 500, "bf16x3", 0), (64, 500, 10009, "bf16x3", 0),
                                              (130, 10501, 10303, "bf16x3", 0)])
def test_gradients(d, N, M, proj, shift):
    prob = W.tiny(d=d, N=N, M=M, P=320, kernel="gauss", kparam=1.1 * np.sqrt(2 * d), n_ft=128, seed=d)
    with QSPlan(d, "gauss", 320, 128, prob.R, prob.kparam, dirs=prob.xi, proj=proj, max_n=N, max_m=M) as plan:
        assert plan.lanes(N) == (N > 1000) and plan.lanes(M) == (M > 1000)
    _check(prob, proj, shift=shift)


@pytest.mark.parametrize("weights", ["none", "one", "tiny", "tiniest", "mixed", "zeros"])
def test_weights(weights):
    import torch

    prob = W.tiny(d=5, N=34000, M=32000, P=320, kernel="laplace", kparam=0.6, n_ft=256, seed=4)
    if weights == "none":
        prob.w = None
    elif weights == "one":  # one weight outweighs all others: the windows' conversions leave the fast range
        prob.w[77] = 1e6
    elif weights == "tiny":
        prob.w *= np.float32(1e-30)
    elif weights == "tiniest":  # the grid's scale is close to the largest number: no finer windows
        prob.w *= np.float32(3e-34)
    elif weights == "mixed":
        prob.w *= np.exp(np.random.default_rng(3).uniform(-12, 0, prob.N)).astype(np.float32)
    with QSPlan(5, "laplace", prob.P, prob.n_ft, prob.R, prob.kparam, dirs=prob.xi, proj="fp32", max_n=prob.N, max_m=prob.M) as plan:
        assert plan.lanes(prob.N) and plan.lanes(prob.M)
        if weights == "zeros":
            s = plan.sum(torch.from_numpy(prob.x).cuda(), torch.zeros(prob.N, device="cuda"), torch.from_numpy(prob.y).cuda())
            plan.check()
            assert not s.any()
            return
    _check(prob, "fp32")


@pytest.mark.parametrize("proj", ["fp32_fused", "fp32", "bf16x3", "tf32"])
def test_data_errors_are_flagged(proj):
    import torch

    prob = W.tiny(d=16, N=34000, M=32000, P=320, kernel="gauss", kparam=6.0, n_ft=256, seed=6)
    data = {"x": torch.from_numpy(prob.x).cuda(), "w": torch.from_numpy(prob.w).cuda(), "y": torch.from_numpy(prob.y).cuda()}
    with QSPlan(16, "gauss", 320, 256, prob.R, prob.kparam, dirs=prob.xi, proj=proj, max_n=prob.N, max_m=prob.M) as plan:
        assert plan.lanes(prob.N) and plan.lanes(prob.M)
        good = plan.sum(**data)
        plan.check()
        for bad, status in ((float("nan"), 3), (float("inf"), 3), (1e4, 2)):
            for which in ("x", "y") if status == 2 else ("x", "y", "w"):
                a = {k: v.clone() for k, v in data.items()}
                a[which].view(-1)[4321] = bad
                plan.sum(**a)
                assert plan.status() == status, (which, bad)
        assert torch.equal(plan.sum(**data), good)  # a failed call leaves nothing behind
        plan.check()


@pytest.mark.parametrize("N,M,bits", [(12001, 12007, True), (12001, 500, True), (500, 12007, True), (12001, 220000, False)])
def test_noalloc(N, M, bits):
    # the last: partial sums without low parts, which are all that fit beside the grids
    import torch

    prob = _problem(6, N, M, 288, 512, N + M)
    x, w, y = (torch.from_numpy(a).cuda() for a in (prob.x, prob.w, prob.y))
    with QSPlan(6, "gauss", 288, 512, prob.R, prob.kparam, dirs=prob.xi, proj="fp32_fused", max_n=N, max_m=M) as plan:
        assert plan.lanes(N) == (N > 1000) and plan.lanes(M) == (M > 1000)
        ref = plan.sum(x, w, y)
        plan.check()
    lib, desc, dirs = _lib.load(), _desc(prob), torch.from_numpy(prob.xi).cuda()
    for _ in range(2):
        out = torch.full((M,), float("nan"), device="cuda")
        assert lib.qs_sum_noalloc(ctypes.byref(desc), dirs.data_ptr(), x.data_ptr(), N, w.data_ptr(), y.data_ptr(), M, out.data_ptr(),
                                  torch.cuda.current_stream().cuda_stream) == 0, lib.qs_last_error().decode()
        if bits:
            assert torch.equal(out, ref)
        else:  # nine groups' sums rounded to FP32
            assert float((out - ref).norm() / ref.norm()) < 1e-6


def test_more_slices_than_low_parts_are_kept_for():
    # P > 2048: the partial buffer holds the groups' sums without their low parts
    import torch

    prob = _problem(3, 2003, 2011, 2200, 128, 5)
    with QSPlan(3, "gauss", 2200, 128, prob.R, prob.kparam, dirs=prob.xi, proj="fp32_fused", max_n=2100, max_m=2100) as plan:
        assert plan.lanes(prob.N) and plan.lanes(prob.M)
        s = plan.sum(*(torch.from_numpy(a).cuda() for a in (prob.x, prob.w, prob.y))).cpu().numpy()
        plan.check()
    assert np.sqrt(np.mean((s - _reference(prob)) ** 2)) < _bound(prob, "fp32", True)
