"""The workloads whose speed is watched, each as a program that uses the package would call it.

``listed()`` gives the named cases, ``draw(rng)`` another one of the same ranges, ``prepare(case, seed)`` what the
program holds before the call (inputs on the GPU and the plan it keeps), ``run(state)`` one pass through the public
entry points, ``work(case)`` the bytes and operations that a pass cannot do without, and ``exact(case, seed)`` the
same outputs from plain torch in 64 bits.

What a case computes is fixed by its "call":

  sum     QSPlan.sum: s_m = sum_n w_n F(|x_n - y_m|) on the device
  train   KernelSumFn: the sum and its gradients in x, w and y through autograd
  grad_y  QSPlan.grad in the targets only: one step of an MMD gradient flow
  host    QSPlan.sum_host: inputs in pinned host memory, result on the host
  sorted  QSPlan.sum_sorted: the negative-distance sum by sorting, without Fourier truncation
  batch   QSBatch.sum: many independent problems in one call
"""
import math

import numpy as np
import torch

from paper_2410_01316_gb300 import KernelSumFn, QSBatch, QSPlan

# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
# "data": ball (uniform in the unit ball), normal (N(0, I)), pca (independent coordinates of decaying variance),
#         sparse (80 % zeros, else U(0, 1)), flow (fixed points ~ N(0, I) and moving ones ~ U[-2, 2]^d)
# "weights": signed (N(0, 1): interpolation and regression coefficients), mean (1 / N: densities, potentials,
#         energy distances), none (the entry point's default of unit weights), flow (the two signs of an MMD flow)


def _case(name, call, d, N, M, P, n_ft, kernel, data, weights, window_kind="es"):
    return {"name": name, "call": call, "d": d, "N": N, "M": M, "P": P, "n_ft": n_ft, "kernel": kernel, "data": data,
            "weights": weights, "window_kind": window_kind}


def listed():
    return [
        # the smallest call: a kernel interpolant evaluated at a thousand points in space, where launches count
        _case("sum_small_d3", "sum", 3, 1000, 1000, 64, 256, "gauss", "ball", "signed", "kb"),
        # a training step of a small point-cloud model in space: forward, and gradients in everything
        _case("train_small_d3", "train", 3, 2048, 1500, 100, 256, "gauss", "normal", "signed"),
        # kernel density of tabular data (d = 16): a training set of odd size against a test set
        _case("sum_tabular_d16", "sum", 16, 15003, 4997, 640, 512, "matern", "normal", "mean"),
        # an image data set in full dimension, the benchmark's headline workload
        _case("sum_images_d784", "sum", 784, 60000, 60000, 2048, 1024, "laplace", "sparse", "mean"),
        # the potential of an energy distance between two large clouds (tensor-core projection, large grid)
        _case("sum_energy_d64", "sum", 64, 200000, 200000, 1024, 2048, "negdist", "normal", "mean"),
        # principal components of a large data set summed against itself, unit weights: the largest number of points
        _case("sum_pca_d30", "sum", 30, 960000, 960000, 1280, 128, "gauss", "pca", "none"),
        # one step of an MMD gradient flow (d = 16): gradients in the particles only
        _case("grad_flow_d16", "grad_y", 16, 200000, 100000, 1024, 1024, "negdist", "flow", "flow"),
        # a training step on embeddings (d = 64): forward, and gradients in sources, weights and targets
        _case("train_embed_d64", "train", 64, 30011, 9973, 512, 512, "gauss", "normal", "mean"),
        # the same in full image dimension, a smaller set
        _case("train_images_d784", "train", 784, 10007, 5003, 1000, 1024, "laplace", "sparse", "mean"),
        # the sum without Fourier truncation, by sorting
        _case("sorted_d64", "sorted", 64, 200000, 200000, 128, 2048, "negdist", "normal", "mean"),
        # inputs that arrive from the host on every call
        _case("host_images_d784", "host", 784, 30001, 29999, 1024, 1024, "laplace", "sparse", "mean"),
        # many independent problems of uneven size in one call (N and M up to the values given)
        _case("batch_48", "batch", 0, 30000, 30000, 256, 512, "gauss", "normal", "signed"),
    ]


# per kernel the numbers of Fourier coefficients that are used with it
_N_FT = {"gauss": (128, 256, 512), "matern": (512,), "laplace": (1024,), "negdist": (512, 1024, 2048)}


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["sum", "sum", "sum", "sum", "train", "train", "grad_y", "sorted", "host", "batch"])
    if call == "batch":
        top = _log_int(rng, 3000, 40000)
        return _drawn("batch", 0, top, top, rng.choice([128, 256]), 512, "gauss", "normal", "signed")
    d = rng.choice([3, 3, 5, 16, 16, 30, 40, 64, 64, 200, 784])
    if call == "grad_y":
        d = rng.choice([3, 16, 16, 30, 64])
        M = _log_int(rng, 1000, 100000)
        P, n_ft = _log_int(rng, 64, 1024), rng.choice([512, 1024])
        return _drawn("grad_y", d, 2 * M, M, P, n_ft, "negdist", "flow", "flow")
    if call == "sorted":
        d = rng.choice([3, 16, 64])
        return _drawn("sorted", d, _log_int(rng, 2000, 200000), _log_int(rng, 2000, 200000), rng.choice([64, 100, 128]),
                      1024, "negdist", "normal", "mean")
    kernel = rng.choice(["gauss", "matern", "laplace", "negdist"])
    n_ft = rng.choice(_N_FT[kernel])
    top = {3: 200000, 5: 200000, 16: 200000, 30: 400000, 40: 200000, 64: 200000, 200: 100000, 784: 60000}[d]
    if call == "train":
        top = min(top, 30000)
    if call == "host":
        top = min(top, 60000)
    N, M, P = _log_int(rng, 1000, top), _log_int(rng, 1000, top), _log_int(rng, 64, 2048)
    P = max(64, min(P, int(8e8 / (N + M))))
    data = "sparse" if d >= 200 else "pca" if d >= 30 and rng.random() < 0.5 else "ball" if d == 3 else "normal"
    weights = rng.choice(["mean", "none"]) if kernel == "negdist" or d > 16 else rng.choice(["mean", "none", "signed"])
    if call == "train":
        weights = "mean" if weights == "none" else weights
    return _drawn(call, d, N, M, P, n_ft, kernel, data, weights, rng.choice(["es", "es", "kb"]))


def _drawn(*a):
    c = _case("", *a)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _directions(d, P, seed):
    """Spherical Fibonacci points in d = 3, else the first P rows of seeded orthogonal matrices."""
    if d == 3:
        p = np.arange(P, dtype=np.float64)
        z = 1.0 - (2.0 * p + 1.0) / P
        phi = 2.0 * math.pi * p / (0.5 * (1.0 + math.sqrt(5.0)))
        r = np.sqrt(np.maximum(0.0, 1.0 - z * z))
        return np.stack([r * np.cos(phi), r * np.sin(phi), z], axis=1).astype(np.float32)
    rng = np.random.default_rng(seed)
    blocks = [np.linalg.qr(rng.standard_normal((d, d)))[0] for _ in range((P + d - 1) // d)]
    return np.ascontiguousarray(np.concatenate(blocks)[:P].astype(np.float32))


def _points(g, data, n, d):
    dev = "cuda"
    if data == "ball":
        x = torch.randn(n, d, generator=g, device=dev)
        r = torch.rand(n, 1, generator=g, device=dev) ** (1.0 / d)
        return x / x.norm(dim=1, keepdim=True) * r
    if data == "pca":
        sd = torch.arange(1, d + 1, device=dev, dtype=torch.float32) ** -0.5
        return torch.randn(n, d, generator=g, device=dev) * sd
    if data == "sparse":
        x = torch.rand(n, d, generator=g, device=dev)
        keep = torch.rand(n, d, generator=g, device=dev) >= 0.8
        return x * keep
    return torch.randn(n, d, generator=g, device=dev)


def _inputs(case, seed):
    """x, w, y, v on the GPU and the parameters that a program derives from them, from the seed alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    N, M, d = case["N"], case["M"], case["d"]
    if case["data"] == "flow":
        # moving particles y first, then the fixed points: the sources of a flow step are both
        y = (torch.rand(M, d, generator=g, device="cuda") * 4.0 - 2.0).contiguous()
        x = torch.cat([y, torch.randn(N - M, d, generator=g, device="cuda")]).contiguous()
    else:
        x = _points(g, case["data"], N, d).contiguous()
        # a data set summed against itself where the sizes are those of one set
        y = x if case["data"] == "pca" and N == M else _points(g, case["data"], M, d).contiguous()
    if case["weights"] == "signed":
        w = torch.randn(N, generator=g, device="cuda")
    elif case["weights"] == "mean":
        w = torch.full((N,), 1.0 / N, device="cuda")
    elif case["weights"] == "flow":
        w = torch.cat([torch.full((M,), 1.0 / M, device="cuda"), torch.full((N - M,), -1.0 / (N - M), device="cuda")])
    else:
        w = None
    v = torch.randn(M, generator=g, device="cuda") / math.sqrt(M)
    # median rule on a thousand pairs, and the radius that bounds the projections
    k = min(1000, N, M)
    i = torch.randint(0, N, (k,), generator=g, device="cuda")
    j = torch.randint(0, M, (k,), generator=g, device="cuda")
    med = float((x[i].double() - y[j].double()).norm(dim=1).median())
    R = float(x.double().norm(dim=1).max() + y.double().norm(dim=1).max()) * (1 + 1e-6)
    kparam = {"gauss": med, "matern": med, "laplace": 1.0 / med, "negdist": 0.0}[case["kernel"]]
    return {"x": x, "w": w, "y": y, "v": v, "R": R, "kparam": kparam, "xi": _directions(d, case["P"], seed)}


def _problems(case):
    """The problems of a batch: d in {3, 16, 64}, N and M spread over two decades (log-uniform), N_ft uneven too."""
    out = []
    for i in range(48):
        N, M = (int(case["N"] * 100.0 ** -math.modf(i * a)[0]) for a in (0.6180339887498949, 0.4142135623730951))
        out.append(dict(case, d=(3, 16, 64)[i % 3], N=N, M=M, n_ft=(256, 512, 1024)[i // 3 % 3]))
    return out


def _plan(case, p):
    nu = 1.5 if case["kernel"] == "matern" else 0.0
    return QSPlan(case["d"], case["kernel"], case["P"], case["n_ft"], p["R"], p["kparam"], dirs=p["xi"],
                  max_n=case["N"], max_m=case["M"], kparam2=nu, window_kind=case["window_kind"])


def prepare(case, seed):
    if case["call"] == "batch":
        subs = [(c, _inputs(c, seed + 1000 * i)) for i, c in enumerate(_problems(case))]
        plans = [_plan(c, p) for c, p in subs]
        batch = QSBatch(plans)
        # the mode that the library's tuner picks for batches of this kind
        batch.set_mode(concurrent=True)
        outs = [torch.empty(c["M"], device="cuda") for c, _ in subs]
        return {"call": "batch", "plans": plans, "batch": batch, "outs": outs,
                "problems": [(p["x"], p["w"], p["y"], o) for (_, p), o in zip(subs, outs)]}
    p = _inputs(case, seed)
    state = {"call": case["call"], "plan": _plan(case, p)}
    if case["call"] == "host":
        for k in ("x", "w", "y"):
            state[k] = None if p[k] is None else p[k].cpu().pin_memory().numpy()
        return state
    for k in ("x", "w", "y", "v"):
        state[k] = p[k]
    if case["call"] == "train":
        for k in ("x", "w", "y"):
            state[k] = state[k].detach().clone().requires_grad_(True)
    return state


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    call = state["call"]
    if call == "sum":
        return state["plan"].sum(state["x"], state["w"], state["y"])
    if call == "train":
        x, w, y = state["x"], state["w"], state["y"]
        s = KernelSumFn.apply(x, w, y, state["plan"])
        gx, gw, gy = torch.autograd.grad(s, (x, w, y), state["v"])
        return {"s": s.detach(), "x": gx, "w": gw, "y": gy}
    if call == "grad_y":
        return state["plan"].grad(state["x"], state["w"], state["y"], None, want=("y",))["y"]
    if call == "host":
        return state["plan"].sum_host(state["x"], state["w"], state["y"])
    if call == "sorted":
        return state["plan"].sum_sorted(state["x"], state["w"], state["y"])
    state["batch"].sum(state["problems"])
    return state["outs"]


def work(case):
    """Points, weights and directions read once, results written once; 2 d operations for each projection of a point
    onto a direction, the window's taps at both ends, and the two transforms of each slice's grid."""
    if case["call"] == "batch":
        subs = [work(dict(c, call="sum")) for c in _problems(case)]
        return {k: sum(o[k] for o in subs) for k in ("bytes", "flops")}
    N, M, d, P, n_ft = (case[k] for k in ("N", "M", "d", "P", "n_ft"))
    b = 4 * ((N + M) * d + N + M + P * d)
    per_slice = (N + M) * (2 * d + 2 * 8) + 2 * 2.5 * 2 * n_ft * math.log2(2 * n_ft)
    f = P * per_slice
    if case["call"] == "sorted":
        f = P * (N + M) * (2 * d + 4)
    if case["call"] == "grad_y":
        b += 4 * M * d
        f += P * M * 2 * d
    if case["call"] == "train":
        # backward: spreads of both sides again, derivative and plain values at both, back-projections
        b += 4 * ((N + M) * d + N + M)
        f += P * per_slice + P * (N + M) * 2 * d + P * N * 16
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# 64 bits
# ---------------------------------------------------------------------------
def _tau(case, p):
    kp, R = p["kparam"], p["R"]
    return {"gauss": lambda: min(0.3 / R, 0.1 / kp), "matern": lambda: min(0.2 / R, 0.1 / kp),
            "laplace": lambda: min(0.1 / R, 0.1 * kp), "negdist": lambda: 0.5 / R}[case["kernel"]]()


def _coefficients(case, p, tau):
    """c_k = tau f^(tau k) for k = 0 .. N_ft / 2, f^(w) = pi^(d/2) / Gamma(d/2) |w|^(d-1) F^(|w|); the triangle wave
    of the negative distance in closed form."""
    d, kp = case["d"], p["kparam"]
    k = np.arange(case["n_ft"] // 2 + 1, dtype=np.float64)
    lg = math.lgamma
    if case["kernel"] == "negdist":
        amp = math.exp(0.5 * math.log(math.pi) + lg(0.5 * (d + 1)) - lg(0.5 * d)) / tau
        c = np.where(k % 2 == 1, amp / (math.pi**2 * np.maximum(k, 1.0) ** 2), 0.0)
        c[0] = -0.25 * amp
        return c
    w = tau * k[1:]
    log_w = (d - 1) * np.log(w)
    lpi = math.log(math.pi)
    if case["kernel"] == "gauss":
        q = 2.0 * math.pi**2 * kp**2 * w**2
        lf = 0.5 * math.log(2.0) + lpi + math.log(kp) + 0.5 * (d - 1) * np.log(q) - q - lg(0.5 * d)
    elif case["kernel"] == "laplace":
        lf = (lg(0.5 * (d + 1)) + d * math.log(2.0) + (d - 0.5) * lpi + log_w - lg(0.5 * d) - d * math.log(kp)
              - 0.5 * (d + 1) * np.log1p(4.0 * math.pi**2 * w**2 / kp**2))
    else:
        nu = 1.5
        lf = (lg(nu + 0.5 * d) + 0.5 * d * math.log(2.0) + d * lpi + d * math.log(kp) + log_w - lg(0.5 * d) - lg(nu)
              - 0.5 * d * math.log(nu) - (nu + 0.5 * d) * np.log1p(2.0 * math.pi**2 * kp**2 * w**2 / nu))
    return np.concatenate([[0.0], tau * np.exp(lf)])  # d > 1 in every case: c_0 = 0


def _powers(a, q, sign):
    """z^0 .. z^(q-1) with z = e^(sign 2 pi i a), by doubling: a (..., n) -> (..., n, q)."""
    z = torch.polar(torch.ones_like(a), sign * 2.0 * math.pi * a).unsqueeze(-1)
    e = torch.ones_like(z)
    while e.shape[-1] < q:
        e = torch.cat([e, e * z], dim=-1)
        z = z * z
    return e[..., :q]


def _spectrum(a, w, nk):
    """sum_n w_n e^(-2 pi i k a_n) for k = 0 .. nk - 1, one row per slice of a (slices, n): k = k1 + q k2."""
    q = 1 << max(0, math.ceil(math.log2(math.sqrt(nk))))
    r = -(-nk // q)
    out = torch.zeros(a.shape[0], r * q, dtype=torch.complex128, device=a.device)
    for part in range(0, a.shape[1], 100000):
        ap, wp = a[:, part:part + 100000], w[part:part + 100000]
        lo = _powers(ap, q, -1.0) * wp[None, :, None]
        hi = _powers(ap * q, r, -1.0)
        out += torch.matmul(hi.transpose(1, 2), lo).reshape(a.shape[0], r * q)
    return out[:, :nk]


def _evaluate(b, h):
    """Re sum_k h_k e^(2 pi i k b_m), one row per slice: b (slices, m), h (slices, nk)."""
    nk = h.shape[1]
    q = 1 << max(0, math.ceil(math.log2(math.sqrt(nk))))
    r = -(-nk // q)
    h = torch.cat([h, h.new_zeros(h.shape[0], r * q - nk)], dim=1).reshape(-1, r, q)
    out = torch.empty_like(b)
    for part in range(0, b.shape[1], 100000):
        bp = b[:, part:part + 100000]
        t = torch.matmul(_powers(bp * q, r, 1.0), h)
        out[:, part:part + 100000] = (t * _powers(bp, q, 1.0)).real.sum(-1)
    return out


def _sliced(case, p, sources, weights, targets, plain, deriv):
    """sum over slices at the targets: (1/P) sum_p t_p and (tau/P) sum_p t'_p xi_p, as far as asked for."""
    P, tau = case["P"], _tau(case, p)
    c = torch.from_numpy(_coefficients(case, p, tau)).cuda()
    k = torch.arange(c.numel(), dtype=torch.float64, device="cuda")
    fac = torch.full_like(c, 2.0)
    fac[0] = fac[-1] = 1.0  # k = 0, and the unpaired k = -N_ft / 2
    xi = torch.from_numpy(p["xi"]).double().cuda()
    X, Y = sources.double(), targets.double()
    w = torch.ones(X.shape[0], dtype=torch.float64, device="cuda") if weights is None else weights.double()
    s = torch.zeros(Y.shape[0], dtype=torch.float64, device="cuda") if plain else None
    g = torch.zeros_like(Y) if deriv else None
    step = max(1, min(P, int(1.5e6 / max(min(100000, X.shape[0]), min(100000, Y.shape[0])))))
    for j in range(0, P, step):
        x = xi[j:j + step]
        h = _spectrum(tau * (x @ X.T), w, c.numel()) * (c * fac)
        b = tau * (x @ Y.T)
        if plain:
            s += _evaluate(b, h).sum(0) / P
        if deriv:
            g += (tau / P) * (_evaluate(b, h * (2j * math.pi * k)).T @ x)
    return s, g


def _sorted_sum(case, p):
    """(1/P) sum_p sum_n w_n f(|a_n - b_m|), f(t) = -c_d |t|, from sorted projections and prefix sums."""
    d, P = case["d"], case["P"]
    cd = math.exp(0.5 * math.log(math.pi) + math.lgamma(0.5 * (d + 1)) - math.lgamma(0.5 * d))
    xi = torch.from_numpy(p["xi"]).double().cuda()
    X, Y, w = p["x"].double(), p["y"].double(), p["w"].double()
    s = torch.zeros(Y.shape[0], dtype=torch.float64, device="cuda")
    zero = torch.zeros(1, dtype=torch.float64, device="cuda")
    for x in xi:
        a, order = torch.sort(X @ x)
        ws = w[order]
        W, S = torch.cat([zero, ws.cumsum(0)]), torch.cat([zero, (ws * a).cumsum(0)])
        b = Y @ x
        i = torch.searchsorted(a, b)
        s += b * (2 * W[i] - W[-1]) - (2 * S[i] - S[-1])
    return s * (-cd / P)


def exact(case, seed):
    if case["call"] == "batch":
        subs = [(c, _inputs(c, seed + 1000 * i)) for i, c in enumerate(_problems(case))]
        return [_sliced(c, p, p["x"], p["w"], p["y"], True, False)[0] for c, p in subs]
    p = _inputs(case, seed)
    if case["call"] == "sorted":
        return _sorted_sum(case, p)
    if case["call"] == "grad_y":
        return _sliced(case, p, p["x"], p["w"], p["y"], False, True)[1]
    if case["call"] == "train":
        s, gy = _sliced(case, p, p["x"], p["w"], p["y"], True, True)
        gw, gx = _sliced(case, p, p["y"], p["v"], p["x"], True, True)
        return {"s": s, "x": gx * p["w"].double()[:, None], "w": gw, "y": gy * p["v"].double()[:, None]}
    s = _sliced(case, p, p["x"], p["w"], p["y"], True, False)[0]
    return s.cpu().numpy() if case["call"] == "host" else s
