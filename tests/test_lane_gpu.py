"""The slice-per-lane grid stages (sums and gradients of at least 2 to 6 million (point, slice) pairs).

Every branch of their dispatch against the FP64 oracle: coordinates per lane (d = 1 .. 64) or projections
from the tensor cores, polynomials or plain cells per window, several windows per slice, points outside the
window, slice counts that fill the last group or not, ragged sizes, unaligned inputs, weights that need the
slow conversion.  Bound, relative to sum|w| max|F| (and its analogue for the gradients): window aliasing and
fit 3e-7, FP32 projections and transform 3e-6 (see test_transform_gpu.py), the rounding of the windows
2^-17 of the edge taps' share (1e-7): 4e-6; BF16x3 projections carry 2^-16 of |u| instead of 2^-24, and the
derivative of the value in u is at most D1 / G: the projection bar of 1e-5 of the other tests.
"""
import numpy as np
import pytest

import oracle
from paper_2410_01316_gb300 import QSPlan
from paper_2410_01316_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": 4e-6, "fp32_fused": 4e-6, "bf16x3": 1e-5, "auto": 4e-6}


def _cuda(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _norms(prob, v):
    t = oracle.tau(prob.kernel, prob.kparam, prob.R)
    c = oracle.coeffs(prob.kernel, prob.kparam, prob.d, t, prob.n_ft)
    k = np.arange(-prob.n_ft // 2, prob.n_ft // 2)
    D1 = float(np.sum(np.abs(2 * np.pi * k * c)))
    maxF = prob.R if prob.kernel == "negdist" else 1.0
    return t, c, D1, maxF


def _check(prob, proj, grads=True, plan_kw=None, shift=0):
    import torch

    v = np.random.default_rng(5).standard_normal(prob.M).astype(np.float32)
    x, y = _cuda(prob.x), _cuda(prob.y)
    if shift:  # the same rows at an address that is 4-byte aligned only
        def unaligned(a):
            buf = torch.empty(a.numel() + shift, device="cuda")
            buf[shift:] = a.reshape(-1)
            return buf[shift:].reshape(a.shape)

        x, y = unaligned(x), unaligned(y)
    w = None if prob.w is None else _cuda(prob.w)
    with QSPlan(prob.d, prob.kernel, prob.P, prob.n_ft, prob.R, prob.kparam, dirs=prob.xi, proj=proj,
                max_n=prob.N, max_m=prob.M, **(plan_kw or {})) as plan:
        s = plan.sum(x, w, y).cpu().numpy().astype(np.float64)
        again = plan.sum(x, w, y).cpu().numpy().astype(np.float64)
        g = plan.grad(x, w, y, _cuda(v)) if grads else {}
        plan.check()
        g = {k: t.cpu().numpy().astype(np.float64) for k, t in g.items()}
    assert np.array_equal(s, again)
    t, c, D1, maxF = _norms(prob, v)
    ww = np.ones(prob.N, np.float32) if prob.w is None else prob.w
    sw, mw = float(np.abs(ww).sum()), float(np.abs(ww).max())
    sv, mv = float(np.abs(v).sum()), float(np.abs(v).max())
    rng = np.random.default_rng(8)
    im, jn = rng.choice(prob.M, 60, replace=False), rng.choice(prob.N, 60, replace=False)
    # the last targets and sources too (remainders of blocks)
    im[:3], jn[:3] = prob.M - 1 - np.arange(3), prob.N - 1 - np.arange(3)
    ref = oracle.o1_sum(prob.x, prob.w, prob.y[im], prob.xi, t, c)
    tol = TOL[proj]
    assert np.max(np.abs(s[im] - ref)) / (sw * maxF) < tol
    if grads:
        rg = oracle.o1_grad(prob.x, prob.w, prob.y, v, prob.xi, t, c, idx_n=jn, idx_m=im)
        assert np.max(np.abs(g["y"][im] - rg["y"])) / (t * sw * mv * D1) < tol
        assert np.max(np.abs(g["x"][jn] - rg["x"])) / (t * mw * sv * D1) < tol
        assert np.max(np.abs(g["w"][jn] - rg["w"])) / (sv * maxF) < tol


@pytest.mark.parametrize("d,P,N,M,proj", [(1, 33, 64003, 63777, "fp32_fused"), (3, 100, 20983, 21001, "auto"),
                                          (4, 64, 32768, 32775, "fp32"), (5, 96, 33003, 34001, "fp32"),
                                          (16, 130, 26001, 24311, "fp32"), (30, 100, 63000, 62999, "fp32"),
                                          (20, 192, 33001, 33003, "fp32"), (40, 128, 50400, 50387, "fp32"), (64, 65, 98001, 97001, "fp32"),
                                          (64, 200, 10501, 10503, "bf16x3"), (100, 97, 22003, 21703, "bf16x3"),
                                          (300, 64, 33001, 32801, "bf16x3")])
def test_dimensions_and_ragged_sizes(d, P, N, M, proj):
    prob = W.tiny(d=d, N=N, M=M, P=P, kernel="gauss", kparam=1.1 * np.sqrt(2 * d), n_ft=128, seed=d + P)
    _check(prob, proj)


@pytest.mark.parametrize("n_ft,P,N", [(256, 70, 90000), (1024, 66, 96000), (2048, 64, 99000)])
@pytest.mark.parametrize("proj", ["fp32_fused", "bf16x3"])
def test_wide_windows_and_several_per_slice(n_ft, P, N, proj):
    # negative distance in d = 40 with one set nearly filling the radius along two axes, so that its
    # projections span most of the period where those of sets within R / 2 would span far less
    d = 40 if proj == "bf16x3" else 32
    prob = W.tiny(d=d, N=N, M=N + 13, P=P, kernel="negdist", kparam=0.0, n_ft=n_ft, seed=n_ft)
    prob.x[:, :2] *= 100.0
    prob.y *= 0.05
    prob.xi[:, 2:] *= 0.02
    prob.xi /= np.linalg.norm(prob.xi, axis=1, keepdims=True)
    if n_ft >= 1024:  # both directions: targets wide, too
        prob.x, prob.y = prob.y[:N].copy(), np.concatenate([prob.x, prob.x[:13]])
    prob.R = W.radius(prob.x, prob.y)
    _check(prob, proj)


@pytest.mark.parametrize("proj", ["fp32", "bf16x3"])
def test_points_outside_the_sampled_window(proj):
    # most points in a narrow cluster, a few far out that a sample of 256 mostly misses
    prob = W.tiny(d=16, N=46000, M=46200, P=70, kernel="gauss", kparam=3.0, n_ft=512, seed=9)
    for a in (prob.x, prob.y):
        a *= 0.1
        a[np.random.default_rng(3).choice(len(a), 25, replace=False)] *= 60.0
    prob.R = W.radius(prob.x, prob.y)
    _check(prob, proj)


@pytest.mark.parametrize("weights", ["none", "one", "tiny", "tiniest", "zeros", "mixed"])
def test_weights(weights):
    prob = W.tiny(d=5, N=34000, M=32000, P=100, kernel="laplace", kparam=0.6, n_ft=256, seed=4)
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
    else:
        import torch

        with QSPlan(5, "laplace", prob.P, prob.n_ft, prob.R, prob.kparam, dirs=prob.xi, max_n=prob.N,
                    max_m=prob.M) as plan:
            s = plan.sum(_cuda(prob.x), torch.zeros(prob.N, device="cuda"), _cuda(prob.y))
            plan.check()
            assert not s.any()
        return
    _check(prob, "fp32")


@pytest.mark.parametrize("d", [3, 4, 6, 16, 30])
def test_unaligned_inputs(d):
    prob = W.tiny(d=d, N=32001, M=32003, P=200 if d > 16 else 100, kernel="gauss", kparam=2.0 * np.sqrt(d), n_ft=128, seed=d)
    _check(prob, "fp32", shift=1)


@pytest.mark.parametrize("proj", ["fp32_fused", "fp32", "bf16x3"])
def test_data_errors_are_flagged(proj):
    import torch

    prob = W.tiny(d=16, N=34000, M=32000, P=100, kernel="gauss", kparam=6.0, n_ft=256, seed=6)
    x, w, y = _cuda(prob.x), _cuda(prob.w), _cuda(prob.y)
    with QSPlan(16, "gauss", prob.P, prob.n_ft, prob.R, prob.kparam, dirs=prob.xi, proj=proj, max_n=prob.N,
                max_m=prob.M) as plan:
        good = plan.sum(x, w, y)
        plan.check()
        for bad, status in ((float("nan"), 3), (float("inf"), 3), (1e4, 2)):
            for which in ("x", "y", "w"):
                if which == "w" and status == 2:
                    continue
                a = {"x": x, "w": w, "y": y}
                a[which] = a[which].clone()
                a[which].view(-1)[4321] = bad
                plan.sum(a["x"], a["w"], a["y"])
                assert plan.status() == status, (which, bad)
        assert torch.equal(plan.sum(x, w, y), good)  # a failed call leaves nothing behind
        plan.check()
