"""What a user of the solver has it do, as cases that can be timed and checked.

The framework solves the scattering system A(h, N) u = rhs on an n^3 grid: its
work is the operator (`Plan.matvec32`, `Plan.matvec`), the solves built on it
(`Plan.solve`, `Plan.solve_batch`, the one-call `solve`), the gradient
(`solve_autograd`) and the field off the grid (`Plan.field`).  Every case calls
one of these as a program does, on seeded draws h ~ U[0.5, 1.5] + i U[0.5, 1.5],
N ~ U[0.5, 1.5] (the repository's input recipe), on the unit cube.

A solve to 1e-6 hands its solution on in complex64 (it has no more digits);
the other solves run to 1e-10 and keep complex128.
"""

from __future__ import annotations

import math

import torch

import paper_1602_04691_gb300 as ori
from paper_1602_04691_gb300 import Plan, inputs

DEV = "cuda"
C_S = 4.0 * math.pi


def listed():
    return [
        # one FP64 operator call on the smallest documented grid: latency and launches only
        {"name": "matvec-fp64-12", "kind": "matvec", "precision": "fp64", "n": 12, "k": 1.0},
        # the FP32 operator a user's own iteration applies: a ragged small grid, a ragged
        # large one (260 needs twice the padding of 256) and the headline size
        {"name": "matvec32-100", "kind": "matvec32", "n": 100, "k": 3.0},
        {"name": "matvec32-260", "kind": "matvec32", "n": 260, "k": 3.0},
        {"name": "matvec32-512", "kind": "matvec32", "n": 512, "k": 5.0},
        # the FP64-class operator in paired FP32, and in native FP64: residual checks
        {"name": "matvec-df-200", "kind": "matvec", "precision": "df", "n": 200, "k": 3.0},
        {"name": "matvec-fp64-130", "kind": "matvec", "precision": "fp64", "n": 130, "k": 2.0},
        # a small solve, the (RED) grid of the numerical experiment: launches and host reads
        {"name": "solve-20", "kind": "solve", "n": 20, "k": 1.0, "tol": 1e-10},
        # the headline solve
        {"name": "solve-512", "kind": "solve", "n": 512, "k": 5.0, "tol": 1e-6},
        # multi-frequency, multi-direction data of the inverse problem: 64 systems in one batch
        {"name": "batch-128", "kind": "batch", "n": 128, "nk": 4, "ndir": 16, "tol": 1e-6},
        # one gradient step: forward solve, misfit on 1024 cells, adjoint solve
        {"name": "grad-128", "kind": "grad", "n": 128, "k": 2.0, "tol": 1e-11},
        # the one-call form: plan, solve, free
        {"name": "oneshot-64", "kind": "oneshot", "n": 64, "k": 2.0, "tol": 1e-10},
        # the scattered field at sensor points, on the (IE) grid of the experiment
        {"name": "field-40", "kind": "field", "n": 40, "k": 1.0, "points": 1000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matvec32", "matvec32", "matvec32", "df", "fp64", "solve", "solve", "batch", "grad",
                       "oneshot", "field"])
    k = round(rng.uniform(0.5, 6.0), 3)
    if kind == "matvec32":
        return {"kind": "matvec32", "n": _log(rng, 8, 512), "k": k}
    if kind == "df":
        return {"kind": "matvec", "precision": "df", "n": _log(rng, 8, 400), "k": k}
    if kind == "fp64":
        return {"kind": "matvec", "precision": "fp64", "n": _log(rng, 8, 200), "k": k}
    if kind == "solve":
        return {"kind": "solve", "n": _log(rng, 8, 400), "k": k, "tol": rng.choice([1e-6, 1e-10])}
    if kind == "batch":
        return {"kind": "batch", "n": _log(rng, 8, 110), "nk": rng.randint(1, 4), "ndir": rng.randint(1, 16),
                "tol": 1e-6}
    if kind == "grad":
        return {"kind": "grad", "n": _log(rng, 8, 200), "k": k, "tol": 1e-11}
    if kind == "oneshot":
        return {"kind": "oneshot", "n": _log(rng, 8, 128), "k": k, "tol": 1e-10}
    return {"kind": "field", "n": _log(rng, 8, 64), "k": k, "points": _log(rng, 16, 2000)}


# -- inputs ---------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _uniform(g, m):
    return torch.rand(m, generator=g, device=DEV, dtype=torch.float64) + 0.5


def _medium(g, m):
    h = torch.complex(_uniform(g, m), _uniform(g, m))
    return h, _uniform(g, m)


def _normal(g, m, dtype):
    return torch.randn(m, generator=g, device=DEV, dtype=dtype)


def _wave_numbers(case):
    return [1.0, 2.0, 4.0, 8.0][:case["nk"]] if case["kind"] == "batch" else [case["k"]]


def _directions(case):
    return [tuple(float(c) for c in a) for a in inputs.fibonacci_directions(case["ndir"])]


def _inputs(case, seed):
    """Everything the case draws, in one order, for prepare() and exact()."""
    g = _gen(seed)
    n, kind = case["n"], case["kind"]
    m = n ** 3
    h, N = _medium(g, m)
    d = {"h": h, "N": N}
    if kind == "matvec32":
        d["x"] = _normal(g, m, torch.complex64)
    elif kind == "matvec":
        d["x"] = _normal(g, m, torch.complex128)
    elif kind == "grad":
        count = min(1024, m // 8)
        d["cells"] = torch.randperm(m, generator=g, device=DEV)[:count]
        d["target"] = _normal(g, count, torch.complex128)
    elif kind == "field":
        d["u"] = _normal(g, m, torch.complex128)
        # sensors in and around the cube
        d["points"] = torch.rand(case["points"], 3, generator=g, device=DEV, dtype=torch.float64) * 3.0 - 1.0
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    state = {"case": case, **d}
    if kind == "oneshot":
        return state
    ks = _wave_numbers(case)
    state["plan"] = Plan(case["n"], ks if kind == "batch" else ks[0], d["h"], d["N"])
    if kind == "grad":
        state["h"].requires_grad_(True)
        state["N"].requires_grad_(True)
    elif kind == "batch":
        state["alphas"] = _directions(case)
    if kind not in ("grad",):
        del state["h"], state["N"]     # the plan keeps its own copy
    return state


def _kept(u, tol):
    return u.to(torch.complex64) if tol >= 1e-6 else u


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "matvec32":
        return state["plan"].matvec32(state["x"], form="B")
    if kind == "matvec":
        return state["plan"].matvec(state["x"], form="A", precision=case["precision"])
    if kind == "solve":
        return _kept(state["plan"].solve(tol=case["tol"])[0], case["tol"])
    if kind == "batch":
        return _kept(state["plan"].solve_batch(state["alphas"], tol=case["tol"])[0], case["tol"])
    if kind == "grad":
        h, N = state["h"], state["N"]
        h.grad = N.grad = None
        u = ori.solve_autograd(state["plan"], h, N, tol=case["tol"])
        miss = u[state["cells"]] - state["target"]
        loss = (miss.real ** 2 + miss.imag ** 2).sum()
        loss.backward()
        return u.detach(), h.grad, N.grad
    if kind == "oneshot":
        return _kept(ori.solve(state["h"], state["N"], case["k"], tol=case["tol"])[0], case["tol"])
    return state["plan"].field(state["u"], state["points"], alpha=(0.0, 0.0, 1.0))


# -- what one pass cannot do without -----------------------------------------------

def _operator_flops(n):
    """One convolution by zero-padded FFTs of 2n points per axis: n^2 lines along x, 2n^2
    along y and 4n^2 along z, forward and inverse (5 m log2 m each), and the product."""
    m = 2 * n
    return 2 * 7 * n * n * 5.0 * m * math.log2(m) + 6.0 * m ** 3


def work(case):
    n, kind = case["n"], case["kind"]
    m = n ** 3
    spec = (n + 1) ** 3                  # distinct entries of the even spectrum
    if kind == "matvec32":
        return {"bytes": 8.0 * (3 * m + spec), "flops": _operator_flops(n)}
    if kind == "matvec":
        return {"bytes": 16.0 * (3 * m + spec), "flops": _operator_flops(n)}
    # COCG gains about half a digit an iteration on these media
    its = 2 * round(-math.log10(case["tol"])) if "tol" in case else 0
    if kind in ("solve", "oneshot"):
        return {"bytes": (16.0 if kind == "solve" else 24.0) * m + 16.0 * m, "flops": its * _operator_flops(n)}
    if kind == "batch":
        r = case["nk"] * case["ndir"]
        return {"bytes": 16.0 * m + 8.0 * m * r, "flops": r * its * _operator_flops(n)}
    if kind == "grad":
        return {"bytes": 24.0 * m + 40.0 * m, "flops": 2 * its * _operator_flops(n)}
    return {"bytes": 40.0 * m + 40.0 * case["points"], "flops": 40.0 * m * case["points"]}


# -- the same results in 64 bits by plain torch ----------------------------------------

class _Operator:
    """K v = c_S |Delta| sum_{p != q} G(x_q, x_p) v_p by FFTs of m = 2n points per axis."""

    def __init__(self, n, k):
        self.n, m = n, 2 * n
        i = torch.arange(m, device=DEV)
        s = torch.minimum(i, m - i).to(torch.float64) / n
        r = (s[:, None, None] ** 2 + s[None, :, None] ** 2 + s[None, None, :] ** 2).sqrt_()
        r[0, 0, 0] = 1.0
        g = torch.polar(1.0 / (4.0 * math.pi * r), k * r)
        del r
        g[0, 0, 0] = 0.0
        for dim in range(3):
            g = torch.fft.fft(g, dim=dim)
        self.g = g.mul_(C_S / n ** 3)

    def __call__(self, v):
        n, m = self.n, 2 * self.n
        t = v.view(n, n, n)
        for dim in (2, 1, 0):
            t = torch.fft.fft(t, n=m, dim=dim)
        t.mul_(self.g)
        for dim in (0, 1, 2):
            t = torch.fft.ifft(t, dim=dim).narrow(dim, 0, n)
        return t.reshape(-1)


def _cocg(K, S, b, tol=1e-13, maxit=80):
    """w with (I + S K S) w = b, by COCG."""
    w = torch.zeros_like(b)
    r, p = b.clone(), b.clone()
    rho, bn = (r * r).sum(), float(b.norm())
    for _ in range(maxit):
        q = p + S * K(S * p)
        a = rho / (p * q).sum()
        w += a * p
        r -= a * q
        if float(r.norm()) <= tol * bn:
            break
        new = (r * r).sum()
        p = r + (new / rho) * p
        rho = new
    return w


def _plane_wave(n, k, a):
    c = (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) / n
    norm = math.sqrt(sum(v * v for v in a))
    e = [torch.polar(torch.ones_like(c), k * v / norm * c) for v in a]
    return (e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]).reshape(-1)


def exact(case, seed):
    d = _inputs(case, seed)
    n, kind = case["n"], case["kind"]
    h, N = d["h"], d["N"]
    w = h * N
    if kind == "field":
        return _exact_field(d, n, case["k"])
    S = w.sqrt()
    if kind == "batch":
        out = []
        for k in _wave_numbers(case):
            K = _Operator(n, k)
            out.append(torch.stack([_cocg(K, S, S * _plane_wave(n, k, a), 1e-11) / S for a in _directions(case)]))
        return torch.stack(out)
    K = _Operator(n, case["k"])
    if kind == "matvec32":
        x = d["x"].to(torch.complex128)
        return x + S * K(S * x)
    if kind == "matvec":
        return d["x"] + K(w * d["x"])
    u = _cocg(K, S, S * _plane_wave(n, case["k"], (0.0, 0.0, 1.0)), 1e-10 if case["tol"] >= 1e-6 else 1e-13) / S
    if kind != "grad":
        return u
    e = torch.zeros_like(u)
    e[d["cells"]] = u[d["cells"]] - d["target"]
    ec = e.conj().resolve_conj()
    t = (ec - S * _cocg(K, S, ec / S)) * u
    return u, (-2.0 * (t / h)).conj().resolve_conj(), -2.0 * t.real / N


def _exact_field(d, n, k):
    c = (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) / n
    z, y, x = torch.meshgrid(c, c, c, indexing="ij")
    cells = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], dim=1)
    Q = -(C_S / n ** 3) * d["h"] * d["N"] * d["u"]
    pts = d["points"]
    out = torch.polar(torch.ones_like(pts[:, 2]), k * pts[:, 2])
    step = max(1, (1 << 26) // cells.shape[0])
    for i in range(0, pts.shape[0], step):
        r = ((pts[i:i + step, None, :] - cells[None, :, :]) ** 2).sum(-1).sqrt_()
        out[i:i + step] += torch.polar(1.0 / (4.0 * math.pi * r), k * r) @ Q
    return out
