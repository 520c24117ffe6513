"""The buffer of the tensor-core back-projection: taken by the first gradient, also under stream capture,
and done without where it does not fit."""
import numpy as np
import pytest

from paper_2410_01316_gb300 import QSPlan

pytestmark = pytest.mark.gpu

D, P, N, M = 64, 1024, 1000, 300032  # projections: 1229 MB
BUFFER = P // 32 * M * 64


def _inputs():
    import torch

    gen = torch.Generator(device="cuda").manual_seed(7)
    x, y = (torch.randn(n, D, generator=gen, device="cuda") for n in (N, M))
    xi = np.random.default_rng(1).standard_normal((P, D))
    xi = (xi / np.linalg.norm(xi, axis=1, keepdims=True)).astype(np.float32)
    return x, y, torch.full((N,), 1.0 / N, device="cuda"), xi, float(x.norm(dim=1).max() + y.norm(dim=1).max()) * 1.01


def _plan(xi, R):
    return QSPlan(D, "gauss", P, 256, R, 11.0, dirs=xi, max_n=N, max_m=M, proj="bf16x3")


def _free():
    import torch

    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_only_gradients_take_it_and_it_may_not_fit():
    import torch

    x, y, w, xi, R = _inputs()
    with _plan(xi, R) as plan:
        assert plan.lanes(M)
        plan.sum(x, w, y)
        before = _free()
        g = plan.grad(x, w, y, None, want=("y",))["y"]
        taken = before - _free()
        assert 0.9 * BUFFER < taken - g.numel() * 4 < 1.1 * BUFFER + (8 << 20)
        assert torch.equal(g, plan.grad(x, w, y, None, want=("y",))["y"])
        plan.check()
    with _plan(xi, R) as plan:
        filler = torch.empty(_free() - BUFFER // 2, dtype=torch.uint8, device="cuda")
        out = plan.grad(x, w, y, None, want=("y",))["y"]
        plan.check()
        del filler
        _free()
        # not tried again: a plan's gradients do not change their bits on the way
        assert torch.equal(out, plan.grad(x, w, y, None, want=("y",))["y"])
        s = plan.sum(x, w, y)
        plan.check()
        assert torch.isfinite(s).all()
    # both within 1e-5 of the exact gradient (the projections' bar), so within 2e-5 of each other
    assert float((out - g).norm() / g.norm()) < 2e-5


def test_first_gradient_under_capture():
    import torch

    x, y, w, xi, R = _inputs()
    with _plan(xi, R) as plan:
        ref = plan.grad(x, w, y, None, want=("x", "w", "y"))
        plan.check()
    with _plan(xi, R) as plan:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            out = plan.grad(x, w, y, None, want=("x", "w", "y"))
        for _ in range(2):
            graph.replay()
        torch.cuda.synchronize()
        for k in ref:
            assert torch.equal(out[k], ref[k]), k
        plan.check()
