"""The sum over slices of the tensor-core back-projection: compensated, and right in every tile.

Coordinates are multiples of 2^-8 of at most 16 bits, directions have at most 8 bits (one BF16 number: the product of
two low parts, which BF16x3 leaves out, is zero) and G tau is a power of two, so that projections are exact in every form and the FP32 and BF16x3 forms of a plan form the same derivative values, bit for bit.  Their
gradients then differ by their back-projections only.  The FP32 one sums chunks of 16 slices by TwoSum; with
compensated sums on both sides the RMS difference is the rounding to FP32 of two results and of the chunks'
products, at most 2^-23 of the RMS result (an uncompensated sum over slices whose additions truncate is 1.8e-7 off).
Against 64 bits every element is compared, for one tile and several, tile widths 16 to 128, a remainder of
components, a last group of slices that is not full and targets that do not fill the last tile: 2e-6 of the largest,
ten times what is left of the rounding of the values.
"""
import math

import pytest

from paper_2410_01316_gb300 import QSPlan

pytestmark = pytest.mark.gpu


def _grad64(x, w, y, xi, R, n_ft):
    """Gradient in y of the sliced negative-distance sums, in 64 bits on the GPU."""
    import torch

    d, P, t = x.shape[1], xi.shape[0], 0.5 / R
    k = torch.arange(1, n_ft // 2 + 1, 2, dtype=torch.float64, device="cuda")
    amp = math.exp(0.5 * math.log(math.pi) + math.lgamma(0.5 * (d + 1)) - math.lgamma(0.5 * d)) / t
    c = 2 * amp / (math.pi * k) ** 2
    g = torch.zeros(y.shape, dtype=torch.float64, device="cuda")
    X, Y, W, D = x.double(), y.double(), w.double(), xi.double()
    for p in range(P):
        a, b = 2 * math.pi * t * (X @ D[p]), 2 * math.pi * t * (Y @ D[p])
        ph = k[:, None] * a[None, :]
        hr, hi = c * (torch.cos(ph) @ W), -c * (torch.sin(ph) @ W)
        q = torch.empty_like(b)
        for m in range(0, len(b), 8192):
            ph = b[m:m + 8192, None] * k[None, :]
            q[m:m + 8192] = -(torch.sin(ph) @ (hr * k)) - torch.cos(ph) @ (hi * k)
        g += (2 * math.pi * t / P) * q[:, None] * D[p]
    return g


def _inputs(d, P, M, seed):
    import torch

    gen = torch.Generator(device="cuda").manual_seed(1000 * seed + d)
    x, y = ((torch.randn(n, d, generator=gen, device="cuda") * (2 / d**0.5) * 256).round() / 256 for n in (900, M))
    step = 2.0 ** -int(math.log2(256 * d**0.5 / 6))  # 6 standard deviations in 8 bits
    xi = (torch.randn(P, d, generator=gen, device="cuda") / d**0.5 / step).round() * step
    assert float(xi.abs().max()) < 256 * step
    return x, torch.full((900,), 1.0 / 1024, device="cuda"), y, xi


def _grad(x, w, y, xi, proj):
    with QSPlan(x.shape[1], "negdist", len(xi), 512, 16.0, 0.0, dirs=xi.cpu().numpy(), proj=proj, max_n=len(y),
                max_m=len(y)) as plan:
        assert plan.lanes(len(y)) and not plan.lanes(900)
        g = plan.grad(x, w, y, None, want=("y",))["y"].double()
        plan.check()
    return g


@pytest.mark.parametrize("d,P", [(16, 1024), (48, 1000), (64, 2048)])
def test_sum_over_slices_is_compensated(d, P):
    x, w, y, xi = _inputs(d, P, 7003, 0)
    a, b = _grad(x, w, y, xi, "bf16x3"), _grad(x, w, y, xi, "fp32")
    assert float((a - b).norm() / b.norm()) < 2.0**-23


@pytest.mark.parametrize("d,P,M", [(64, 1024, 5003), (72, 1000, 5003), (130, 1024, 5120), (200, 600, 6001), (784, 513, 7000)])
def test_every_tile_against_64_bits(d, P, M):
    x, w, y, xi = _inputs(d, P, M, 1)
    ref = _grad64(x, w, y, xi, 16.0, 512)
    assert float((_grad(x, w, y, xi, "bf16x3") - ref).abs().max()) < 2e-6 * float(ref.abs().max())


def test_tf32_and_bf16x3_give_the_same_bits_from_the_same_projections():
    import torch

    x, w, y, xi = _inputs(64, 1000, 7003, 2)  # 11 bits hold every coordinate
    assert torch.equal(_grad(x, w, y, xi, "tf32"), _grad(x, w, y, xi, "bf16x3"))
