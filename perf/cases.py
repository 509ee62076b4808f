"""Timed cases of the library: what a program that uses it has it do.

A case is one pass of one kind of call (``op``) at one size:

* ``solve``     far field of a few incidences on a factored contrast (hs_solve, host arrays);
* ``forward``   hs_build of a contrast, then far field and total fields of a batch (hs_forward_dev);
* ``jacobian``  hs_build, then the Jacobian in device memory (hs_jacobian_dev);
* ``gradient``  misfit and gradient through torch.autograd (autograd.misfit: build, forward, adjoint);
* ``gn``        hs_build and a Gauss-Newton step from the normal equations (hs_gn_step);
* ``lsqr``      hs_build and a Gauss-Newton step by LSQR with FP64 products (hs_gn_step_lsqr);
* ``sweep``     recursive_linearization over a few frequencies: new k, new tree, new context.

Sizes follow the sweep plans of the package (plan_ceil: S = 1.6 k, M = P = 4 k, leaves
2^ceil(log2(0.8 k)); plan_c5: twice as many leaves per side) and the benchmark's workloads.
Contrasts are smooth random sine series; measured data are the Born approximation of such a
contrast plus 1% noise, so that they depend on the seed alone.

``exact`` solves the same discrete problem (Chebyshev leaves, flux continuity, Green's identity
on the boundary, Nystrom with product integration) by one dense system on the leaf edges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1608_06871_gb300 as hs
from paper_1608_06871_gb300.autograd import misfit
from paper_1608_06871_gb300.sweep import plan_ceil, recursive_linearization, square_safe

R = 3.0
FP64, MIXED = "fp64", "mixed"


def _case(name, op, k, leaves, S1, S2, M, P, precision, **more):
    c = {"op": op, "k": float(k), "leaves": leaves, "S1": S1, "S2": S2, "M": M, "P": P, "precision": precision,
         "bm_eta": 0.0, "leaf_impedance": False}
    if name is not None:
        c["name"] = name
    c.update(more)
    return c


def listed():
    return [
        # one more incidence on a small factored contrast: the smallest call, all latency
        _case("solve_k5_fp64", "solve", 5.0, 4, 10, 10, 1, 32, FP64),
        # a handful of incidences on a mid-size factored contrast (refinement, few columns)
        _case("solve_k20_mixed", "solve", 20.0, 16, 32, 32, 5, 81, MIXED),
        # one Newton step at the bottom of a sweep: 4 x 4 leaves, 100 unknowns
        _case("gn_k5_fp64", "gn", 5.0, 4, 10, 10, 16, 32, FP64),
        # the first frequencies of a reconstruction: every step a new k, trees 4 x 4 and 8 x 8
        _case("sweep_k2_8_mixed", "sweep", 2.0, 0, 0, 0, 0, 0, MIXED, step=1.0, count=7),
        # combined-field exterior rows and impedance leaves (resonance-free options), odd sizes
        _case("forward_k10_combined_mixed", "forward", 10.0, 8, 16, 13, 37, 61, MIXED, bm_eta=1.0, leaf_impedance=True),
        # misfit gradient for a descent method at 1600 unknowns, through autograd
        _case("gradient_k20_fp64", "gradient", 20.0, 16, 40, 40, 64, 128, FP64),
        # explicit Jacobian in the middle of the k = 1..40 sweep
        _case("jacobian_k20_mixed", "jacobian", 20.0, 16, 32, 32, 80, 80, MIXED),
        # the paper's own step (LSQR at 1e-3) at the same frequency, stopped early: without
        # reorthogonalisation later iterates follow the rounding
        _case("lsqr_k20_mixed", "lsqr", 20.0, 16, 32, 32, 80, 80, MIXED),
        # forward batch of the paper-scale plan at half its top frequency: 64 x 64 leaves
        _case("forward_k35_mixed", "forward", 35.0, 64, 70, 70, 140, 140, MIXED),
        # the benchmark's forward batch, both precisions
        _case("forward_k40_mixed", "forward", 40.0, 32, 40, 40, 128, 256, MIXED),
        _case("forward_k40_fp64", "forward", 40.0, 32, 40, 40, 128, 256, FP64),
        # one Newton step at the top of the k = 1..40 sweep: 4096 unknowns, 160 x 160 data
        _case("gn_k40_mixed", "gn", 40.0, 32, 64, 64, 160, 160, MIXED),
    ]


def draw(rng):
    op = rng.choice(["solve", "forward", "forward", "forward", "jacobian", "gradient", "gn", "lsqr", "sweep"])
    precision = rng.choice([FP64, MIXED, MIXED])
    opts = {"bm_eta": rng.choice([0.0, 0.0, 0.0, 1.0]), "leaf_impedance": rng.random() < 0.2}
    if op == "sweep":
        return _case(None, op, round(rng.uniform(1.5, 3.0), 2), 0, 0, 0, 0, 0, precision,
                     step=round(rng.uniform(0.5, 1.2), 2), count=rng.randint(3, 6))
    top = 40.0 if op in ("solve", "forward") else 24.0
    k = math.exp(rng.uniform(math.log(2.0), math.log(top)))
    # off the square's Dirichlet eigenvalues, as the sweep plans do (Green's rows are singular there)
    k = square_safe(k, near=0.01, window=0.05, unit=math.pi / 2.0)
    leaves = plan_ceil(k).leaves_per_side
    if op == "forward" and precision == MIXED and rng.random() < 0.3:
        leaves *= 2
    S1, S2 = (max(2, int(rng.uniform(0.7, 1.7) * k)) for _ in range(2))
    if op == "solve":
        M, P = int(math.exp(rng.uniform(0.0, math.log(24.0)))), max(3, int(rng.uniform(1.0, 5.0) * k))
    else:
        M, P = (max(3, int(rng.uniform(1.5, 4.0) * k)) for _ in range(2))
    return _case(None, op, k, leaves, S1, S2, M, P, precision, **opts)


# ---- inputs ---------------------------------------------------------------------------------
def _coefficients(S1, S2, rng, qmax=0.3, decay=8.0):
    """Coefficients of a smooth random contrast, max |q| = qmax on a 257 x 257 sample."""
    m1, m2 = np.arange(1.0, S1 + 1), np.arange(1.0, S2 + 1)
    c = rng.standard_normal((S1, S2)) * np.exp(-np.hypot(m1[:, None], m2[None, :]) / decay)
    t = np.linspace(0.0, 1.0, 257)
    q = np.sin(math.pi * np.outer(t, m1)) @ c @ np.sin(math.pi * np.outer(m2, t))
    return c * (qmax / np.max(np.abs(q)))


def _angles(M, P):
    return 2.0 * math.pi * np.arange(M) / M, 2.0 * math.pi * np.arange(P) / P


def _born(c, k, al, th, rng):
    """Measured data: -k^2 int G(x_p, y) q(y) exp(i k d.y) dy with the large-argument Green's
    function, midpoint rule, plus 1% complex noise per incidence."""
    n = max(32, int(math.ceil(4.0 * k)))
    y = (np.arange(n) + 0.5) * (2.0 / n) - 1.0
    s = lambda S: np.sin(0.5 * math.pi * np.outer(y + 1.0, np.arange(1, S + 1)))
    q = (s(c.shape[0]) @ c @ s(c.shape[1]).T).ravel() * (2.0 / n) ** 2
    y1, y2 = np.repeat(y, n), np.tile(y, n)
    r = np.hypot(R * np.cos(th)[:, None] - y1, R * np.sin(th)[:, None] - y2)
    G = 0.25j * np.sqrt(2.0 / (math.pi * k * r)) * np.exp(1j * (k * r - 0.25 * math.pi))
    u = np.exp(1j * k * (np.cos(al)[:, None] * y1 + np.sin(al)[:, None] * y2))
    d = -k * k * (u * q) @ G.T
    e = rng.standard_normal(d.shape) + 1j * rng.standard_normal(d.shape)
    return d + 0.01 * e * (np.linalg.norm(d, axis=1) / np.linalg.norm(e, axis=1))[:, None]


def _inputs(case, seed):
    """Everything of a case that comes from its seed (host arrays)."""
    rng = np.random.default_rng(seed)
    k, op = case["k"], case["op"]
    if op == "sweep":
        plans = [plan_ceil(k + j * case["step"]) for j in range(case["count"])]
        truth = _coefficients(8, 8, rng, qmax=0.05, decay=3.0)
        data = {p.k: _born(truth, p.k, *_angles(p.M, p.P), rng) for p in plans}
        return {"plans": plans, "data": data}
    x = {"c": _coefficients(case["S1"], case["S2"], rng)}
    x["al"], x["th"] = _angles(case["M"], case["P"])
    if op in ("gradient", "gn", "lsqr"):
        x["data"] = _born(x["c"] + 0.2 * _coefficients(case["S1"], case["S2"], rng), k, x["al"], x["th"], rng)
    if op == "lsqr":  # the paper's triangle of modes
        m = np.arange(1, max(case["S1"], case["S2"]) + 1)
        x["mask"] = ((m[:, None] + m[None, :]) <= max(case["S1"], case["S2"]) + 1)[:case["S1"], :case["S2"]]
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    x["case"], op = case, case["op"]
    x["precision"] = hs.HS_MIXED if case["precision"] == MIXED else hs.HS_FP64
    if op == "sweep":
        return x
    dev = torch.device("cuda")
    x["solver"] = hs.Solver(case["leaves"], case["S1"], case["S2"], R, x["precision"], bm_eta=case["bm_eta"],
                            leaf_impedance=case["leaf_impedance"])
    M, P = case["M"], case["P"]
    if op == "solve":
        x["solver"].build(x["c"], case["k"])
    if op in ("forward", "jacobian", "gradient"):
        x["al_d"], x["th_d"] = (torch.tensor(x[a], dtype=torch.float64, device=dev) for a in ("al", "th"))
    if op == "forward":
        x["ufar"] = torch.empty((M, P, 2), dtype=torch.float64, device=dev)
        x["u"] = torch.empty((M, case["leaves"] ** 2, 256, 2), dtype=torch.float64, device=dev)
    if op == "jacobian":
        x["J"] = torch.empty((M * P, case["S1"] * case["S2"], 2), dtype=torch.float64, device=dev)
    if op == "gradient":
        x["data_d"] = torch.view_as_real(torch.tensor(x["data"], device=dev)).contiguous()
        x["c_d"] = torch.tensor(x["c"], device=dev, requires_grad=True)
    return x


def run(x):
    case, op = x["case"], x["case"]["op"]
    if op == "sweep":
        r = recursive_linearization(x["plans"], lambda p, al, th: x["data"][p.k], precision=x["precision"], R=R)
        return {"c": r.c, "residuals": [h["residuals"][0] for h in r.history]}
    s, k = x["solver"], case["k"]
    if op == "solve":
        return s.solve(x["al"], x["th"])
    if op == "forward":
        s.build(x["c"], k)
        hs.hs_forward_dev(s.ctx, x["al_d"], x["th_d"], x["ufar"], x["u"])
        return {"ufar": x["ufar"], "u": x["u"]}
    if op == "jacobian":
        s.build(x["c"], k)
        hs.hs_jacobian_dev(s.ctx, x["al_d"], x["th_d"], x["J"])
        return x["J"]
    if op == "gradient":
        value = misfit(x["c_d"], s, k, x["data_d"], x["al_d"], x["th_d"])
        return {"misfit": value.detach(), "grad": torch.autograd.grad(value, x["c_d"])[0]}
    s.build(x["c"], k)
    if op == "gn":
        c, rn = s.gn_step(x["data"], x["al"], x["th"], 1e-4, x["c"])
        return {"c": c, "resid": rn}
    c, rn, its = s.gn_step_lsqr(x["data"], x["al"], x["th"], x["c"], mask=x["mask"], tol=1e-3, max_iter=10)
    return {"c": c, "resid": rn, "iterations": its}


# ---- what a pass cannot do without ----------------------------------------------------------
def _tree(n):
    """(boxes, interface nodes, parent boundary nodes) of every merge level of n x n leaves."""
    sx = sy = 1
    out = []
    while sx < n or sy < n:
        horiz = sx == sy
        ni = 14 * (sy if horiz else sx)
        sx, sy = (2 * sx, sy) if horiz else (sx, 2 * sy)
        out.append(((n // sx) * (n // sy), ni, 28 * (sx + sy)))
    return out


def _build_flops(n):
    leaf = 2 / 3 * 196 ** 3 + 2 * 196 ** 2 * 56 + 2 * 56 ** 2 * 196 + 8 / 3 * 56 ** 3 + 8 * 56 ** 3 + 4 * 196 * 56 ** 2
    merges = sum(b * (32 / 3 * i ** 3 + 16 * i * i * p + 8 * i * p * p) for b, i, p in _tree(n))
    return n * n * leaf + merges + 32 / 3 * (56 * n) ** 3


def _solve_flops(n, fields):
    """Of one right-hand side: the root system, and the sweep down to the leaves."""
    down = sum(8 * b * 2 * i * p for b, i, p in _tree(n)) + 8 * n * n * 252 * 56
    return 24 * (56 * n) ** 2 + (down if fields else 0)


def _pass_work(op, n, S1, S2, M, P):
    nX, nm, nd = 14 * n, S1 * S2, n * n * 256
    far = 16 * 56 * n * M * P
    by, fl = 8 * (nm + M + P), 0.0
    if op == "solve":
        return {"bytes": 8 * (M + P) + 16 * M * P, "flops": M * _solve_flops(n, False) + far}
    fl += _build_flops(n) + far
    if op == "forward":
        return {"bytes": by + 16 * M * P + 16 * M * nd, "flops": fl + M * _solve_flops(n, True)}
    fl += (M + P) * _solve_flops(n, True)
    contract = 4.0 * M * P * (S1 * nX * nX + nm * nX)
    if op == "jacobian":
        return {"bytes": by + 16 * M * P * nm, "flops": fl + contract}
    by += 16 * M * P + 8 * nm
    if op == "gradient":
        return {"bytes": by, "flops": fl + 8.0 * M * P * nX * nX}
    if op == "gn":
        return {"bytes": by, "flops": fl + contract + 2.0 * M * P * nm * nm + 2 / 3 * nm ** 3}
    return {"bytes": by, "flops": fl + contract + 10.0 * 8 * M * P * nm}  # ten LSQR iterations


def work(case):
    if case["op"] != "sweep":
        return _pass_work(case["op"], case["leaves"], case["S1"], case["S2"], case["M"], case["P"])
    total = {"bytes": 0.0, "flops": 0.0}
    for j in range(case["count"]):
        p = plan_ceil(case["k"] + j * case["step"])
        for key, v in _pass_work("gn", p.leaves_per_side, p.S, p.S, p.M, p.P).items():
            total[key] += v
    return total


# ---- the same discrete problem in plain torch, 64 bits --------------------------------------
def _hankel(x):
    """H_0 and H_1 of the first kind, x > 0: the power series below 2; above, Hankel's integral
    sqrt(2 / (pi x)) exp(i (x - n pi/2 - pi/4)) / Gamma(n + 1/2) int e^(-t^2) t^(2n) (1 + i t^2/(2x))^(n - 1/2) dt
    by the trapezoidal rule, which converges like exp(-2 pi sqrt(x) / step)."""
    z = torch.clamp(x, max=2.0)
    y, log = -0.25 * z * z, torch.log(0.5 * z) + np.euler_gamma
    j0, j1, s0, s1 = (torch.zeros_like(z) for _ in range(4))
    term, harm = torch.ones_like(z), 0.0                         # y^m / m!^2, 1 + 1/2 + ... + 1/m
    for m in range(18):
        j0, s0 = j0 + term, s0 - harm * term
        j1, s1 = j1 + term / (m + 1), s1 + (2.0 * harm + 1.0 / (m + 1)) * term / (m + 1)
        term, harm = term * y / (m + 1) ** 2, harm + 1.0 / (m + 1)
    j1, s1 = 0.5 * z * j1, 0.5 * z * s1
    h0 = torch.complex(j0, (2.0 / math.pi) * (log * j0 + s0))
    h1 = torch.complex(j1, (2.0 / math.pi) * (log * j1 - 0.5 * s1 - 1.0 / z))
    far = x > 2.0
    w = x[far]
    i0, i1 = (torch.zeros(w.shape, dtype=torch.complex128, device=x.device) for _ in range(2))
    for t in np.arange(0, 45) * 0.15:
        root = torch.sqrt(torch.complex(torch.ones_like(w), 0.5 * t * t / w))
        g = (0.15 if t == 0.0 else 0.3) * math.exp(-t * t)
        i0, i1 = i0 + g / root, i1 + g * t * t * root
    front = torch.sqrt(2.0 / (math.pi * w)) / math.sqrt(math.pi) * torch.polar(torch.ones_like(w), w - 0.25 * math.pi)
    h0[far], h1[far] = front * i0, -2.0j * front * i1
    return h0, h1


class _Dense:
    """Leaves eliminated to Dirichlet-to-Neumann maps, one unknown per leaf edge node: flux
    continuity inside, Green's identity (D - I/2) u_s = S d_n u_s on the boundary.  (With the
    combined-field rows the boundary data are the same away from resonances, up to the boundary
    quadrature's error.)"""

    def __init__(self, k, n, c):
        self.k, self.n, self.h = k, n, 2.0 / n
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=self.dev)
        t = -np.cos(math.pi * np.arange(16) / 15)
        D = self._derivative(t) * n          # d/dx on a leaf of width 2 / n
        D2 = D @ D
        self.x = -1.0 + (np.arange(n)[:, None] + 0.5 * (t + 1.0)[None, :]) * self.h  # (n, 16)
        s = lambda S, z: np.sin(0.5 * math.pi * np.outer(np.arange(1, S + 1), z + 1.0))
        q = s(c.shape[0], self.x.ravel()).T @ c @ s(c.shape[1], self.x.ravel())
        q = q.reshape(n, 16, n, 16).transpose(2, 0, 1, 3)[:, :, 1:15, 1:15].reshape(n * n, 196)  # leaf iy n + ix
        r = np.arange(1, 15)
        edge = np.concatenate([r * 16, 240 + r, r * 16 + 15, r])                      # S, E, N, W
        inner = (r[:, None] * 16 + r[None, :]).ravel()
        lap = np.kron(D2, np.eye(16)) + np.kron(np.eye(16), D2)
        dx, dy = np.kron(D, np.eye(16)), np.kron(np.eye(16), D)
        out = np.concatenate([-dy[r * 16], dx[240 + r], dy[r * 16 + 15], -dx[r]])     # outward derivatives
        A = T(lap[np.ix_(inner, inner)])[None] + torch.diag_embed(T(k * k * (1.0 - q)))
        self.LU = torch.linalg.lu_factor(A)
        self.X = torch.linalg.lu_solve(*self.LU, T(lap[np.ix_(inner, edge)])[None].expand(n * n, -1, -1))
        self.Ni = T(out[:, inner])
        dtn = T(out[:, edge])[None] - self.Ni[None] @ self.X
        iy, ix, a = np.arange(n)[:, None, None], np.arange(n)[None, :, None], np.arange(14)
        hor = lambda j, i: n * (n + 1) * 14 + (j * n + i) * 14 + a                    # horizontal line j, column i
        ver = lambda i, j: (i * n + j) * 14 + a                                       # vertical line i, row j
        ids = np.concatenate([hor(iy, ix), ver(ix + 1, iy), hor(iy + 1, ix), ver(ix, iy)], axis=2)
        self.ids = T(ids.reshape(n * n, 56))
        N = 28 * n * (n + 1)
        F = torch.zeros((N, N), dtype=torch.float64, device=self.dev)                 # summed outward fluxes
        F.index_put_((self.ids[:, :, None].expand(-1, 56, 56), self.ids[:, None, :].expand(-1, 56, 56)), dtn,
                     accumulate=True)
        p = np.arange(n)[:, None]
        self.b = T(np.concatenate([v.ravel() for v in (hor(0, p), ver(n, p), hor(n, p), ver(0, p))]))
        self._boundary(t[1:15])
        S, Dl = (T(m) for m in self._layers())
        self.S, self.Au = S, Dl - 0.5 * torch.eye(len(self.b), device=self.dev)
        self.Fb = F[self.b].to(torch.complex128)
        K = F.to(torch.complex128)
        K[self.b] = -self.S @ self.Fb
        K[self.b[:, None], self.b[None, :]] += self.Au
        self.K = torch.linalg.lu_factor(K)
        self.N = N

    @staticmethod
    def _derivative(t):
        d = t[:, None] - t[None, :] + np.eye(len(t))
        w = 1.0 / np.prod(d, axis=1)
        D = w[None, :] / w[:, None] / d
        np.fill_diagonal(D, 0.0)
        return D - np.diag(D.sum(axis=1))

    def _boundary(self, t):
        n, h = self.n, self.h
        z, o = np.zeros(n), np.ones(n)
        g = -1.0 + h * np.arange(n)
        self.p0 = np.concatenate([np.stack(v, 1) for v in ((g, -o), (o, g), (g, o), (-o, g))])
        self.tau = np.concatenate([np.stack(v, 1) for v in ((o, z), (z, o), (o, z), (z, o))])
        self.nu = np.concatenate([np.stack(v, 1) for v in ((z, -o), (o, z), (z, o), (-o, z))])
        self.t = t
        V = np.polynomial.legendre.legvander(t, 13)
        self.w = np.tile(np.linalg.solve(V.T, 2.0 * np.eye(14)[0]) * h / 2.0, 4 * n)
        self.y = (self.p0[:, None] + (0.5 * h * (t + 1.0))[None, :, None] * self.tau[:, None]).reshape(-1, 2)
        self.ny = np.repeat(self.nu, 14, axis=0)

    def _kernels(self, d, ny):
        """G and dG/dn_y for x - y = d (..., 2)."""
        r = np.hypot(d[..., 0], d[..., 1])
        h0, h1 = _hankel(torch.as_tensor(self.k * r, device=self.dev))
        return 0.25j * h0.cpu().numpy(), 0.25j * self.k * h1.cpu().numpy() * (d * ny).sum(-1) / r

    def _layers(self):
        """Single and double layer on the boundary nodes; sources within one panel length by
        Gauss-Legendre graded dyadically toward the target's nearest point."""
        n, h = self.n, self.h
        d = self.y[:, None] - self.y[None, :]
        d[np.arange(len(d)), np.arange(len(d))] = 1.0
        S, Dl = self._kernels(d, self.ny[None])
        S, Dl = S * self.w, Dl * self.w
        gx, gw = np.polynomial.legendre.leggauss(16)
        rules = {}

        def rule(s):  # offsets from s on [0, h], weights, Lagrange basis at the points
            if s not in rules:
                off, wt = [], []
                for end in (-s, h - s):
                    if end != 0.0:
                        e = np.append(end * 0.5 ** np.arange(57), 0.0)
                        off.append((0.5 * (e[1:] + e[:-1])[:, None] + 0.5 * (e[:-1] - e[1:])[:, None] * gx).ravel())
                        wt.append((0.5 * np.abs(e[:-1] - e[1:])[:, None] * gw).ravel())
                off, wt = np.concatenate(off), np.concatenate(wt)
                v = 2.0 * (s + off) / h - 1.0
                L = np.ones((len(v), 14))
                for j in range(14):
                    for l in range(14):
                        if l != j:
                            L[:, j] *= (v - self.t[l]) / (self.t[j] - self.t[l])
                rules[s] = off, wt, L
            return rules[s]

        ends = np.stack([self.p0, self.p0 + h * self.tau], 1)
        for p in range(4 * n):
            for q in range(4 * n):
                u = np.clip(((ends[p] - self.p0[q]) * self.tau[q]).sum(-1), 0.0, h)
                v = np.clip(((ends[q] - self.p0[p]) * self.tau[p]).sum(-1), 0.0, h)
                gap = min(np.min(np.hypot(*(ends[p] - self.p0[q] - u[:, None] * self.tau[q]).T)),
                          np.min(np.hypot(*(ends[q] - self.p0[p] - v[:, None] * self.tau[p]).T)))
                if gap > h * (1.0 + 1e-9):
                    continue
                for i in range(14 * p, 14 * p + 14):
                    s = 0.5 * h * (self.t[i - 14 * p] + 1.0) if p == q else \
                        float(np.clip(np.dot(self.y[i] - self.p0[q], self.tau[q]), 0.0, h))
                    off, wt, L = rule(s)
                    perp = np.zeros(2) if p == q else self.y[i] - (self.p0[q] + s * self.tau[q])
                    g, dg = self._kernels(perp - off[:, None] * self.tau[q], self.nu[q])
                    S[i, 14 * q:14 * q + 14], Dl[i, 14 * q:14 * q + 14] = (g * wt) @ L, (dg * wt) @ L
        return S, Dl

    def _receivers(self, th):
        xp = R * np.stack([np.cos(th), np.sin(th)], 1)
        G, dG = self._kernels(xp[:, None] - self.y[None], self.ny[None])
        return torch.as_tensor(dG * self.w, device=self.dev), torch.as_tensor(-G * self.w, device=self.dev)

    def _grid(self, v):
        """Leaf interiors (leaf, 196, m) as (m, 14 n, 14 n)."""
        return v.reshape(self.n, self.n, 14, 14, -1).permute(4, 1, 2, 0, 3).reshape(-1, 14 * self.n, 14 * self.n)

    def forward(self, al, th):
        """Far field (M, P), fields on the edges (leaf, 56, M) and in the leaves (leaf, 196, M)."""
        d = np.stack([np.cos(al), np.sin(al)])
        ui = np.exp(1j * self.k * (self.y @ d))
        dni = torch.as_tensor(1j * self.k * (self.ny @ d) * ui, device=self.dev)
        ui = torch.as_tensor(ui, device=self.dev)
        rhs = torch.zeros((self.N, len(al)), dtype=torch.complex128, device=self.dev)
        rhs[self.b] = self.Au @ ui - self.S @ dni
        u = torch.linalg.lu_solve(*self.K, rhs)
        Ap, As = self._receivers(th)
        far = (Ap @ (u[self.b] - ui) + As @ (self.Fb @ u - dni)).T
        ue = u[self.ids]
        return far, ue, -(self.X.to(torch.complex128) @ ue)

    def adjoint(self, th):
        """Fields z_p in the leaves with d far(m, p) = sum_x z_p(x) k^2 dq(x) u_m(x) (leaf, 196, P)."""
        Ap, As = self._receivers(th)
        y = As @ self.Fb
        y[:, self.b] += Ap
        y = torch.linalg.lu_solve(*self.K, y.T.conj().resolve_conj().contiguous(), adjoint=True).conj().resolve_conj()
        g = -y
        g[self.b] = self.S.T @ y[self.b] + As.T
        rhs = self.Ni.T.to(torch.complex128)[None] @ g[self.ids]
        both = torch.cat([rhs.real, rhs.imag], dim=-1).contiguous()
        z = torch.linalg.lu_solve(*self.LU, both, adjoint=True)
        return torch.complex(*z.chunk(2, dim=-1))

    def jacobian(self, u, z, S1, S2):
        """J (M P, S1 S2) from leaf fields u and adjoint fields z."""
        s = lambda S: torch.as_tensor(np.sin(0.5 * math.pi * np.outer(np.arange(1, S + 1), self.x[:, 1:15].ravel() + 1)),
                                      dtype=torch.complex128, device=self.dev)
        U, Z, s1, s2 = self._grid(u), self._grid(z), s(S1), s(S2)
        return self.k ** 2 * torch.cat([(s1 @ (U[m] * Z) @ s2.T).reshape(len(Z), S1 * S2) for m in range(len(U))])


def _gn(solver, data, al, th, c):
    """c after one Gauss-Newton step (normal equations, lambda = 1e-4 tr / n) and the residual norm."""
    far, _, u = solver.forward(al, th)
    J = solver.jacobian(u, solver.adjoint(th), *c.shape)
    r = torch.as_tensor(data, device=solver.dev) - far
    A, b = torch.cat([J.real, J.imag]), torch.cat([r.real.ravel(), r.imag.ravel()])
    H = A.T @ A
    H += torch.eye(len(H), dtype=H.dtype, device=H.device) * (1e-4 * torch.trace(H) / len(H))
    dc = torch.linalg.solve(H, A.T @ b)
    return c + dc.cpu().numpy().reshape(c.shape), float(torch.linalg.norm(b))


def _lsqr(A, b, tol, most):
    """Paige and Saunders' LSQR, stopped at a relative residual or normal-equations residual of tol."""
    x = torch.zeros(A.shape[1], dtype=A.dtype, device=A.device)
    beta = first = float(torch.linalg.norm(b))
    u = b / beta
    v = A.T @ u
    alpha = float(torch.linalg.norm(v))
    v = v / alpha
    w, phibar, rhobar, norm2 = v.clone(), beta, alpha, 0.0
    for _ in range(most):
        u = A @ v - alpha * u
        beta = float(torch.linalg.norm(u))
        u = u / beta
        norm2 += alpha * alpha + beta * beta
        v = A.T @ u - beta * v
        alpha = float(torch.linalg.norm(v))
        v = v / alpha
        rho = math.hypot(rhobar, beta)
        c, s = rhobar / rho, beta / rho
        x = x + (c * phibar / rho) * w
        w = v - (s * alpha / rho) * w
        rhobar, phibar = -c * alpha, s * phibar
        if phibar / first <= tol or alpha * abs(c) / math.sqrt(norm2) <= tol:
            break
    return x


def exact(case, seed):
    op = case["op"]
    x = _inputs(case, seed)
    if op == "sweep":
        c, res = np.zeros((1, 1)), []
        for p in x["plans"]:
            if p.leaves_per_side > 8:
                return None
            big = np.zeros((p.S, p.S))
            big[:c.shape[0], :c.shape[1]] = c
            c, rn = _gn(_Dense(p.k, p.leaves_per_side, big), x["data"][p.k], *_angles(p.M, p.P), big)
            res.append(rn)
        return {"c": c, "residuals": res}
    if case["leaves"] > 16:  # a dense system of 30,000 unknowns and more: over 20 seconds
        return None
    s = _Dense(case["k"], case["leaves"], x["c"])
    al, th, c = x["al"], x["th"], x["c"]
    if op == "gn":
        c, rn = _gn(s, x["data"], al, th, c)
        return {"c": c, "resid": rn}
    far, ue, ui = s.forward(al, th)
    if op == "solve":
        return far.cpu().numpy()
    if op == "forward":
        u = torch.zeros((len(al), case["leaves"] ** 2, 16, 16), dtype=torch.complex128, device=s.dev)
        e = ue.permute(2, 0, 1)
        u[:, :, 1:15, 1:15] = ui.permute(2, 0, 1).reshape(len(al), -1, 14, 14)
        u[:, :, 1:15, 0], u[:, :, 15, 1:15], u[:, :, 1:15, 15], u[:, :, 0, 1:15] = e.split(14, dim=2)
        return {"ufar": torch.view_as_real(far.contiguous()), "u": torch.view_as_real(u.reshape(len(al), -1, 256))}
    z = s.adjoint(th)
    J = s.jacobian(ui, z, *c.shape)
    if op == "jacobian":
        return torch.view_as_real(J)
    r = (torch.as_tensor(x["data"], device=s.dev) - far).reshape(-1)
    if op == "gradient":
        return {"misfit": 0.5 * torch.linalg.norm(r) ** 2, "grad": -(J.conj().T @ r).real.reshape(c.shape)}
    keep = torch.as_tensor(x["mask"].ravel(), device=s.dev)
    dc = torch.zeros(c.size, dtype=torch.float64, device=s.dev)
    dc[keep] = _lsqr(torch.cat([J.real, J.imag])[:, keep].contiguous(), torch.cat([r.real, r.imag]), 1e-3, 10)
    return {"c": c + dc.cpu().numpy().reshape(c.shape), "resid": float(torch.linalg.norm(r)), "iterations": None}
