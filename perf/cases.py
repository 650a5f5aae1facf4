"""The workloads whose speed is followed: calls of the library as its users make them.

A case is a problem (mesh, degrees, chaos, coefficient, precisions) and one call on it:

    apply     y = A x, or A^T x (``sg_apply``): the operator by itself, FP64 or double-word
    vcycle    z = P^-1 r (``sg_vcycle``): the preconditioner by itself
    solve     A x = b for one slab (``sg_solve_slab``)
    march     one step in time: right-hand side, solve, mean and variance fields
    mc        mean, variance and paths of a batch of Monte-Carlo samples (``mc_solve_batch``)
    adjoint   E||u(T)||^2 and its gradient in every amplitude and cell (``sg_adjoint_gradient``)

Sizes are those of the workloads in ``inputs`` and of the tests, or lie between them.
``exact`` computes the same outputs in 64 bits with dense element matrices in torch.
"""
import math

import numpy as np
import torch

import paper_2605_21046_gb300 as sg
from paper_2605_21046_gb300 import inputs

MG = {"fp64": sg.SG_PREC_FP64, "fp32": sg.SG_PREC_FP32, "bf16": sg.SG_PREC_BF16}


def _case(kind, dim, nx, ny, nz, k, r, m, p, coef="sine", **more):
    return dict(kind=kind, dim=dim, nx=nx, ny=ny, nz=nz, k=k, r=r, M=m, P=p, coef=coef, **more)


def listed():
    return [
        # the smallest problem, called in a loop by a user's own solver: launches and latency
        dict(_case("apply", 2, 8, 8, 1, 1, 1, 2, 2, prec="fp64"), name="apply q1 8x8"),
        # the ordinary problem, shape tuned once as a long run does
        dict(_case("apply", 2, 64, 64, 1, 2, 1, 4, 3, prec="fp64", tune=True), name="apply q2 64x64"),
        # odd counts of cells, rectangular cells, three time nodes, the adjoint direction
        dict(_case("apply", 2, 45, 37, 1, 2, 2, 3, 2, prec="fp64", trans=True), name="apply q2 45x37 dg2 T"),
        # many modes and a per-cell mean field in double-word arithmetic
        dict(_case("apply", 2, 128, 128, 1, 2, 1, 4, 4, "cells", prec="dw"), name="apply q2 128x128 dw"),
        # the discretisation of the published tables: cubic elements, four time nodes, 11 coefficient terms
        dict(_case("apply", 2, 128, 128, 1, 3, 3, 4, 2, "square", prec="fp64"), name="apply q3 dg3 128x128"),
        # the large 3D problem
        dict(_case("apply", 3, 32, 32, 32, 2, 1, 3, 3, prec="fp64", tune=True), name="apply q2 32x32x32"),
        # the preconditioner by itself, with single-precision and with bf16-stored factors
        dict(_case("vcycle", 2, 64, 64, 1, 2, 1, 4, 3, mg="fp32"), name="vcycle q2 64x64"),
        dict(_case("vcycle", 3, 32, 32, 32, 2, 1, 3, 3, mg="bf16"), name="vcycle q2 32x32x32 bf16"),
        # one step in time of the ordinary problem
        dict(_case("march", 2, 64, 64, 1, 2, 1, 4, 3, prec="fp64", mg="fp32", slabs=100), name="march q2 64x64"),
        # one slab of the large problem with the fastest precision split
        dict(_case("solve", 3, 32, 32, 32, 2, 1, 3, 3, prec="dw", mg="bf16", slabs=20), name="solve q2 32x32x32 dw"),
        # a Monte-Carlo batch over a few slabs
        dict(_case("mc", 2, 32, 32, 1, 2, 1, 4, 3, mg="fp32", slabs=4, samples=256), name="mc q2 32x32"),
        # a gradient for an optimisation loop over the coefficient
        dict(_case("adjoint", 2, 32, 32, 1, 2, 1, 2, 2, "adjoint", prec="fp64", mg="fp32", slabs=8), name="adjoint q2 32x32"),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _modes(m, p):
    return math.comb(m + p, p)


def draw(rng):
    kind = rng.choice(["apply"] * 6 + ["vcycle"] * 2 + ["march", "solve", "mc", "adjoint"])
    while True:
        if kind == "apply":
            if rng.random() < 0.3:
                c = _case(kind, 3, *(_log(rng, 3, 32) for _ in range(3)), rng.choice([1, 2, 2]), rng.choice([0, 1, 1]),
                          rng.randint(1, 4), rng.randint(0, 3))
            else:
                k = rng.choice([1, 2, 2, 3])
                c = _case(kind, 2, _log(rng, 7, 160), _log(rng, 7, 160), 1, k, rng.choice([0, 1, 1, 2, 3]), 4 if k == 3 else
                          rng.randint(1, 4), rng.randint(0, 4 if k < 3 else 2), "square" if k == 3 else rng.choice(["sine", "cells"]))
            c.update(prec=rng.choice(["fp64", "fp64", "dw"]), trans=rng.random() < 0.3)
        elif kind in ("vcycle", "march", "solve"):
            # meshes that coarsen: an even number of cells, halved down to a small odd or even one
            if rng.random() < 0.3:
                n = rng.choice([8, 12, 16, 20, 24, 32])
                c = _case(kind, 3, n, n, n, rng.choice([1, 2]), 1, rng.randint(1, 3), rng.randint(1, 3))
            else:
                c = _case(kind, 2, rng.choice([16, 24, 40, 48, 64, 96]), rng.choice([16, 32, 48, 56, 64]), 1, rng.choice([1, 2, 2]),
                          rng.choice([0, 1, 1, 2]), rng.randint(2, 4), rng.randint(1, 4))
            c.update(mg=rng.choice(["fp32", "bf16"]))
            if kind != "vcycle":
                c.update(prec=rng.choice(["fp64", "dw"]), slabs=rng.choice([10, 20, 50, 100]))
        elif kind == "mc":
            c = _case(kind, 2, rng.choice([16, 24, 32]), rng.choice([16, 32]), 1, rng.choice([1, 2]), 1, rng.randint(2, 4), 2,
                      mg=rng.choice(["fp32", "bf16"]), slabs=rng.randint(2, 4), samples=_log(rng, 33, 256))
        else:
            c = _case(kind, 2, rng.choice([16, 24, 32]), rng.choice([16, 24, 32]), 1, rng.choice([1, 2]), rng.choice([1, 1, 2]), 2,
                      rng.randint(1, 3), "adjoint", prec="fp64", mg="fp32", slabs=rng.randint(3, 8))
        # nothing above the largest listed problem of its kind, and at most 512 modes
        if _modes(c["M"], c["P"]) <= 512 and _unknowns(c) <= 11_000_000 and (c["dim"] == 3 or _unknowns(c) <= 9_300_000):
            return c


# ------------------------------------------------------------------ the problems

def _cells(c):
    return (c["nx"], c["ny"], c["nz"])[: c["dim"]]


def _unknowns(c):
    rows = c["samples"] if c["kind"] == "mc" else _modes(c["M"], c["P"])
    return rows * (c["r"] + 1) * math.prod(c["k"] * n + 1 for n in _cells(c))


def _spec(c, seed):
    """The problem in the format of ``inputs``; a per-cell field comes from the seed."""
    dim, M = c["dim"], c["M"]
    field = np.random.default_rng(seed).uniform(0.8, 1.2, math.prod(_cells(c)))
    lo, slabs = 0.0, c.get("slabs", 100)
    if c["coef"] == "square":
        coef, lo, slabs = inputs.paper_coefficient(), -1.0, 64
    elif c["coef"] == "adjoint":
        coef = inputs.linear_sine_coef(M, dim, 0.1, [(1, 0), (0, 1)] + [(1, 1)] * (M - 2), a0_cells=field)
        coef.insert(1, dict(mu=(0,) * M, amp=0.2, factors=[("pow", 2), ("one", 0)], cell_scale=None))
    else:
        coef = inputs.linear_sine_coef(M, dim, 0.05, [(m,) * dim for m in range(1, M + 1)],
                                       a0_cells=field if c["coef"] == "cells" else None)
    # a Monte-Carlo batch marches to its last slab: slabs of the 50-slab run
    T = 1.0 if c["kind"] not in ("mc", "adjoint") else 0.02 * slabs
    return dict(dim=dim, cells=_cells(c), lo=(lo,) * dim, hi=(1.0,) * dim, k=c["k"], r=c["r"], n_slabs=slabs, T=T, M=M,
                P=c["P"], coef=coef)


def _indices(M, p):
    """Chaos multi-indices of total degree at most p: by degree, then the first variable's degree descending."""
    def of(m, d):
        return [(d,)] if m == 1 else [(a,) + t for a in range(d, -1, -1) for t in of(m - 1, d - a)]
    return [a for d in range(p + 1) for a in of(M, d)]


def _manufactured(c):
    """u = (t + t^2) sum 0.35^|a| prod sin(pi f x) Psi_a, of degree 2 in the chaos."""
    idx = _indices(c["M"], 2)
    return dict(q=2, c=[0.35 ** sum(a) for a in idx],
                freq=[[1 + a[d % c["M"]] % 2 for d in range(c["dim"])] for a in idx], T=[0.0, 1.0, 1.0])


def _interior(c):
    m = torch.ones([c["k"] * n + 1 for n in reversed(_cells(c))], dtype=torch.float64, device="cuda")
    for d in range(m.dim()):
        m.select(d, 0).zero_()
        m.select(d, -1).zero_()
    return m.reshape(-1)


def _random(c, seed, masked):
    """U(-1, 1) per unknown; zero on the boundary where it is a residual or a right-hand side."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.rand(_unknowns(c), dtype=torch.float64, device="cuda", generator=g).mul_(2).sub_(1)
    if masked:
        v.view(-1, _interior(c).numel()).mul_(_interior(c))
    return v


def _samples(c, seed):
    return np.random.default_rng(seed).standard_normal((c["samples"], c["M"]))


# the tolerance at which states are kept for a gradient (the default of the adjoint calls)
RTOL = 1e-10


def prepare(case, seed):
    c = case
    kind = c["kind"]
    ctx = sg.sg_setup_spec(_spec(c, seed), sg.SG_PREC_DW if c.get("prec") == "dw" else sg.SG_PREC_FP64)
    s = dict(case=c, ctx=ctx)
    if c.get("tune"):
        sg.sg_autotune(ctx)
    if kind in ("march", "mc", "adjoint"):
        sg.sg_set_exact(ctx, _manufactured(c))
    if kind in ("vcycle", "solve", "march", "adjoint"):
        sg.sg_mg_setup(ctx, MG[c["mg"]], 1, 0.9)
    if kind in ("apply", "vcycle", "solve"):
        s["x"] = _random(c, seed, kind != "apply")
        s["y"] = torch.empty_like(s["x"])
    elif kind == "march":
        # the state after a slab: smooth in space, so a multiple of the manufactured one plus a small random part
        s["u"] = _previous(c, seed)
        s["rhs"], s["y"] = torch.empty_like(s["u"]), torch.empty_like(s["u"])
        s["mean"], s["var"] = (torch.empty(ctx.info["n_x"], dtype=torch.float64, device="cuda") for _ in range(2))
    elif kind == "mc":
        s["xi"] = _samples(c, seed)
    return s


def run(state):
    s, c, ctx = state, state["case"], state["ctx"]
    kind = c["kind"]
    if kind == "apply":
        sg.sg_apply(ctx, 0, s["x"], s["y"], transpose=c.get("trans", False))
        return s["y"]
    if kind == "vcycle":
        return sg.sg_vcycle(ctx, s["x"], s["y"])
    if kind == "solve":
        s["y"].zero_()
        sg.sg_solve_slab(ctx, 1, s["x"], s["y"], rtol=RTOL)
        return s["y"]
    if kind == "march":
        sg.sg_rhs(ctx, 1, s["u"], s["rhs"])
        s["y"].copy_(s["u"])
        sg.sg_solve_slab(ctx, 1, s["rhs"], s["y"], rtol=RTOL)
        sg.sg_moments(ctx, s["y"], ctx.info["n_t"] - 1, s["mean"], s["var"])
        return {k: s[k] for k in ("rhs", "y", "mean", "var")}
    if kind == "mc":
        mean, var, paths, _ = sg.mc_solve_batch(ctx, s["xi"], batch=64, mg_precision=MG[c["mg"]], rtol=RTOL, keep_paths=True)
        return {"mean": mean, "var": var, "paths": paths}
    J, amp, cell, _ = sg.sg_adjoint_gradient(ctx, rtol=RTOL, checkpoint_every=4, cell_piece=0)
    return {"J": J, "amp": amp, "cell": cell}


# ------------------------------------------------------------------ what a pass cannot do without

def _apply_flops(c, rows, coupled=True):
    """Sum-factorised interpolation and gradients there and back, time-mass coupling, chaos coupling."""
    n, d, nt, cells = c["k"] + 1, c["dim"], c["r"] + 1, math.prod(_cells(c))
    per = 2 * 2 * n * n ** d * d * 2 + 2 * nt * n ** d
    if coupled:
        # nonzeros per row of the coupling: the mean term and, per variable, the neighbours up and down (all products for a square)
        nnz = sum(1 + sum((a[m] > 0) + (sum(a) < c["P"]) for m in range(c["M"])) for a in _indices(c["M"], c["P"])) / rows
        per += 2 * (nnz * (2 if c["coef"] == "square" else 1)) * d * n ** d
    else:
        per += 2 * d * n ** d
    return cells * rows * nt * per


def _vcycle_work(c, rows):
    """nu = 1: two sweeps, two residuals and the transfers of every level (1 + 2^-d + ... of the finest)."""
    n, d, nt, cells = c["k"] + 1, c["dim"], c["r"] + 1, math.prod(_cells(c))
    levels = 1 / (1 - 0.5 ** d)
    np_ = nt * n ** d
    flops = levels * (2 * 2 * cells * np_ * np_ * rows + 2 * _apply_flops(c, rows, False))
    value = {"fp64": 8, "fp32": 4, "bf16": 4}[c["mg"]]
    factor = {"fp64": 8, "fp32": 4, "bf16": 2}[c["mg"]]
    n_u = rows * nt * math.prod(c["k"] * m + 1 for m in _cells(c))
    return {"bytes": 16 * n_u + levels * (cells * np_ * np_ * factor + 4 * n_u * value), "flops": flops}


def _solve_work(c, rows, its, coupled=True):
    n_u = rows * (c["r"] + 1) * math.prod(c["k"] * m + 1 for m in _cells(c))
    v = _vcycle_work(c, rows)
    krylov = sum(4 * (j + 1) + 1 for j in range(its)) * 2 * n_u
    return {"bytes": its * v["bytes"] + 16 * n_u + sum(8 * n_u * (j + 4) for j in range(its)),
            "flops": its * (v["flops"] + _apply_flops(c, rows, coupled)) + krylov}


def work(case):
    c = case
    rows = c["samples"] if c["kind"] == "mc" else _modes(c["M"], c["P"])
    n_u = _unknowns(c)
    if c["kind"] == "apply":
        return {"bytes": 16.0 * n_u, "flops": float(_apply_flops(c, rows))}
    if c["kind"] == "vcycle":
        return _vcycle_work(c, rows)
    its = 11  # about one iteration per digit
    w = _solve_work(c, rows, its, c["kind"] != "mc")
    if c["kind"] == "mc":
        return {k: v * c["slabs"] for k, v in w.items()}
    if c["kind"] == "adjoint":
        return {k: v * 2 * c["slabs"] for k, v in w.items()}
    return {k: float(v) for k, v in w.items()}


# ------------------------------------------------------------------ the same in 64 bits

def _lagrange(nodes, x):
    """Values and derivatives [x][node] of the Lagrange basis."""
    v, dv = np.ones((len(x), len(nodes))), np.zeros((len(x), len(nodes)))
    for i, ni in enumerate(nodes):
        p = np.poly1d([1.0])
        for j, nj in enumerate(nodes):
            if j != i:
                p = p * np.poly1d([1.0, -nj]) / (ni - nj)
        v[:, i], dv[:, i] = p(x), p.deriv()(x)
    return v, dv


def _lobatto(k):
    return np.array({1: [0, 1], 2: [0, 0.5, 1], 3: [0, 0.5 - 0.5 / 5 ** 0.5, 0.5 + 0.5 / 5 ** 0.5, 1]}[k], dtype=np.float64)


def _gauss(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (x + 1), 0.5 * w


def _radau(r):
    """Right Radau points: zeros of P_r - P_{r+1} on [-1, 1], mapped to [0, 1]."""
    c = np.zeros(r + 2)
    c[r], c[r + 1] = 1.0, -1.0
    x = np.sort(np.polynomial.legendre.legroots(c).real)
    x[-1] = 1.0
    return 0.5 * (x + 1)


def _psi(n, y):
    """Orthonormal Hermite polynomial of degree n."""
    return np.polynomial.hermite_e.hermeval(y, [0.0] * n + [1.0]) / math.sqrt(math.factorial(n))


def _pieces(spec):
    coef, M = spec["coef"], spec["M"]
    if not isinstance(coef, dict):
        return coef
    # d_min + (sum xi_m g_m)^2: xi_m^2 = sqrt(2) psi_2 + 1
    one = ("one", 0)
    power = lambda f, g: [("pow", a + b) if a + b else one for (_, a), (_, b) in zip(f, g)]  # noqa: E731
    e = lambda *ms: tuple(sum(m == i for m in ms) for i in range(M))  # noqa: E731
    out = [dict(mu=e(), amp=coef["d_min"], factors=[one, one])]
    for m in range(M):
        for mu, amp in ((e(), 1.0), (e(m, m), math.sqrt(2.0))):
            out.append(dict(mu=mu, amp=amp, factors=power(coef["g"][m], coef["g"][m])))
        out += [dict(mu=e(m, n), amp=2.0, factors=power(coef["g"][m], coef["g"][n])) for n in range(m + 1, M)]
    return out


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


class _Plain:
    """One discretisation: dense reference-element tables, gathered cells."""

    def __init__(self, spec, cells=None, n_gauss=None, diagonal=False, samples=None):
        self.spec, self.dim, self.k = spec, spec["dim"], spec["k"]
        self.cells = tuple(cells or spec["cells"])
        dim, k = self.dim, self.k
        self.h = [(spec["hi"][d] - spec["lo"][d]) / self.cells[d] for d in range(dim)]
        self.nn = [k * n + 1 for n in self.cells]
        self.nodes, self.nt = _lobatto(k), spec["r"] + 1
        xq, wq = _gauss(n_gauss or k + 1)
        S, dS = _lagrange(self.nodes, xq)

        def product(tables):  # x fastest in points and in nodes
            out = tables[0]
            for t in tables[1:]:
                out = np.kron(t, out)
            return out
        self.phi = _t(product([S] * dim))                                      # [point][node]
        self.grad = [_t(product([dS if e == d else S for e in range(dim)]) / self.h[d]) for d in range(dim)]
        self.w = _t(product([wq[None]] * dim)[0] * math.prod(self.h))
        # global node of every local node of every cell
        grid = np.meshgrid(*[np.arange(n) for n in reversed(self.cells)], indexing="ij")
        c = [g.reshape(-1) for g in reversed(grid)]
        a = [g.reshape(-1) for g in reversed(np.meshgrid(*[np.arange(k + 1)] * dim, indexing="ij"))]
        stride = [math.prod(self.nn[:d]) for d in range(dim)]
        self.conn = torch.as_tensor(sum((c[d][:, None] * k + a[d][None]) * stride[d] for d in range(dim)), device="cuda")
        q = [g.reshape(-1) for g in reversed(np.meshgrid(*[xq] * dim, indexing="ij"))]
        self.x = [spec["lo"][d] + self.h[d] * (c[d][:, None] + q[d][None]) for d in range(dim)]
        self.n_x = math.prod(self.nn)
        inner = np.ones([n for n in reversed(self.nn)])
        for d in range(dim):
            np.moveaxis(inner, d, 0)[[0, -1]] = 0.0
        self.inner = _t(inner.reshape(-1))
        # time: mass tau int phi_i phi_j, transport int phi_j' phi_i + phi_j(0) phi_i(0)
        self.tau = spec["T"] / spec["n_slabs"]
        tn = _radau(spec["r"])
        xt, wt = _gauss(self.nt + 2)
        v, dv = _lagrange(tn, xt)
        self.t_nodes, self.v0, self.v1 = tn, _lagrange(tn, np.array([0.0]))[0][0], _lagrange(tn, np.array([1.0]))[0][0]
        self.At = _t(np.einsum("q,qi,qj->ij", wt, v, dv) + np.outer(self.v0, self.v0))
        self.Bt = _t(self.tau * np.einsum("q,qi,qj->ij", wt, v, v))
        self.Ct = _t(np.outer(self.v0, self.v1))
        # coefficient fields of the active terms and the coupling of the rows
        self.pieces = _pieces(spec)
        self.mus = list(dict.fromkeys(tuple(p["mu"]) for p in self.pieces))
        self.a = [0.0] * len(self.mus)
        for p in self.pieces:
            self.a[self.mus.index(tuple(p["mu"]))] += p["amp"] * self.field(p)
        self.a = [_t(f) for f in self.a]
        idx = _indices(spec["M"], spec["P"])
        if samples is not None:
            psi = np.array([[np.prod([_psi(m, x) for m, x in zip(mu, xi)]) for mu in self.mus] for xi in samples])
            self.couple = lambda f: sum(_t(psi[:, t])[:, None, None, None] * a for t, a in enumerate(self.a)) * f
        else:
            G = [_t(_triples(idx, mu, idx)) for mu in self.mus]
            if diagonal:  # the block of the mean term alone
                zero = self.mus.index((0,) * spec["M"])
                self.couple = lambda f: self.a[zero] * f
            else:
                self.G = G
                self.couple = lambda f: sum(a * torch.einsum("ab,bicq->aicq", g, f) for g, a in zip(G, self.a))

    def field(self, piece, scaled=True):
        f = np.ones_like(self.x[0])
        for d, (kind, kk) in enumerate(piece["factors"][: self.dim]):
            f = f * (np.sin(kk * np.pi * self.x[d]) if kind == "sin" else self.x[d] ** kk if kind == "pow" else 1.0)
        s = piece.get("cell_scale")
        if s is None or not scaled:
            return f
        s = np.asarray(s).reshape(tuple(reversed(self.spec["cells"])))
        while s.shape != tuple(reversed(self.cells)):  # children averaged
            for d in range(s.ndim):
                s = s.reshape(s.shape[:d] + (s.shape[d] // 2, 2) + s.shape[d + 1:]).mean(axis=d + 1)
        return f * s.reshape(-1)[:, None]

    def gather(self, u):
        return (u.reshape(-1, self.nt, self.n_x) * self.inner)[:, :, self.conn]

    def scatter(self, y):
        out = torch.zeros(y.shape[0], y.shape[1], self.n_x, dtype=torch.float64, device="cuda")
        out.index_add_(2, self.conn.reshape(-1), y.reshape(y.shape[0], y.shape[1], -1))
        return out * self.inner

    def mass(self, u, Tm):
        """(I x Tm x M) u on the interior."""
        f = torch.einsum("ij,ajcn,qn->aicq", Tm, self.gather(u), self.phi) * self.w
        return self.scatter(f @ self.phi)

    def apply(self, u, trans=False):
        u = u.reshape(-1, self.nt, self.n_x)
        g, At = self.gather(u), self.At.T if trans else self.At
        y = torch.einsum("ij,ajcq->aicq", At, g @ self.phi.T * self.w) @ self.phi
        for gr in self.grad:
            y += torch.einsum("ij,ajcq->aicq", self.Bt, self.couple(g @ gr.T) * self.w) @ gr
        return self.scatter(y) + u * (1 - self.inner)

    # ---- solves: the constant-coefficient operator, inverted by the eigenvectors of its 1D factors, as preconditioner
    def _fast(self):
        if hasattr(self, "Z"):
            return
        self.Z, lam = [], []
        x, w = _gauss(self.k + 1)
        v, dv = _lagrange(self.nodes, x)
        for d in range(self.dim):
            n = self.nn[d]
            M, K = np.zeros((n, n)), np.zeros((n, n))
            for c in range(self.cells[d]):
                s = slice(c * self.k, c * self.k + self.k + 1)
                M[s, s] += self.h[d] * np.einsum("q,qi,qj->ij", w, v, v)
                K[s, s] += np.einsum("q,qi,qj->ij", w, dv, dv) / self.h[d]
            L = np.linalg.inv(np.linalg.cholesky(M[1:-1, 1:-1]))
            ev, Q = np.linalg.eigh(L @ K[1:-1, 1:-1] @ L.T)
            Z = np.zeros((n, n - 2))
            Z[1:-1] = L.T @ Q
            self.Z.append(_t(Z))
            lam.append(ev)
        total = sum(_t(lam[d]).reshape([-1 if e == d else 1 for e in reversed(range(self.dim))]) for d in range(self.dim))
        zero = self.mus.index((0,) * self.spec["M"])
        mean = float((self.a[zero] * self.w).sum() / (self.w.sum() * self.a[zero].shape[0]))
        self.blocks = torch.linalg.inv(self.At + mean * total[..., None, None] * self.Bt)

    def inverse0(self, r, trans):
        self._fast()
        v = r.reshape([-1, self.nt] + list(reversed(self.nn)))
        for d in range(self.dim):
            v = torch.movedim(torch.movedim(v, -1 - d, -1) @ self.Z[d], -1, -1 - d)
        v = torch.einsum("...ji,aj...->ai..." if trans else "...ij,aj...->ai...", self.blocks, v)
        for d in range(self.dim):
            v = torch.movedim(torch.movedim(v, -1 - d, -1) @ self.Z[d].T, -1, -1 - d)
        return v.reshape(-1, self.nt, self.n_x)

    def solve(self, b, trans=False):
        """Corrections by the preconditioner, their images orthogonal to the last ones (GCR)."""
        b = b.reshape(-1, self.nt, self.n_x)
        x, r, past = torch.zeros_like(b), b * self.inner, []
        size = r.norm()
        for _ in range(120):
            if r.norm() <= 3e-15 * size:
                break
            p = self.inverse0(r, trans)
            ap = self.apply(p, trans)
            for q, aq in past:
                f = (ap * aq).sum()
                p, ap = p - f * q, ap - f * aq
            f = 1 / ap.norm()
            p, ap = p * f, ap * f
            past = past[-8:] + [(p, ap)]
            f = (r * ap).sum()
            x, r = x + f * p, r - f * ap
        return x + b * (1 - self.inner)

    # ---- one V-cycle of the mean block (every mode alike)
    def vcycle(self, b, factors, omega):
        b = b.reshape(-1, self.nt, self.n_x)
        x = b * (1 - self.inner)
        n_in = self.nt * int(self.inner.sum())
        if n_in <= 1024 or any(n % 2 or n <= 2 for n in self.cells):
            at = torch.nonzero(self.inner).reshape(-1)
            e = torch.zeros(n_in, self.nt, self.n_x, dtype=torch.float64, device="cuda")
            e[torch.arange(n_in), torch.arange(self.nt).repeat_interleave(at.numel()), at.repeat(self.nt)] = 1.0
            A = self.apply(e)[:, :, at].reshape(n_in, n_in).T
            x[:, :, at] = torch.linalg.solve(A, b[:, :, at].reshape(-1, n_in).T).T.reshape(-1, self.nt, at.numel())
            return x
        inv, count = self._patches(factors), self.scatter(torch.ones(1, 1, *self.conn.shape, dtype=torch.float64, device="cuda")).clamp_(min=1)

        def smooth(x):
            r = self.gather(b - self.apply(x)).permute(2, 1, 3, 0).flatten(1, 2)      # [cell][time, node][row]
            z = (inv @ r).unflatten(1, (self.nt, -1)).permute(3, 1, 0, 2)
            return x + omega * self.scatter(z) / count
        x = smooth(x)
        C = _Plain(self.spec, [n // 2 for n in self.cells], diagonal=True)
        P = []
        for d in range(self.dim):
            m = np.zeros((self.nn[d], C.nn[d]))
            for i in range(self.nn[d]):
                cell = min(i // self.k, self.cells[d] - 1)
                s = 0.5 * (cell + self.nodes[i - cell * self.k])
                cc = min(int(s), C.cells[d] - 1)
                m[i, cc * self.k: cc * self.k + self.k + 1] = _lagrange(self.nodes, np.array([s - cc]))[0][0]
            m[[0, -1]] = 0.0
            m[:, [0, -1]] = 0.0
            P.append(_t(m))

        def move(v, nn, tables):
            v = v.reshape([-1, self.nt] + list(reversed(nn)))
            for d, t in enumerate(tables):
                v = torch.movedim(torch.movedim(v, -1 - d, -1) @ t, -1, -1 - d)
            return v.reshape(v.shape[0], self.nt, -1)
        e = C.vcycle(move(b - self.apply(x), self.nn, P), factors, omega)
        return smooth(x + move(e, C.nn, [t.T for t in P]))

    def _patches(self, factors):
        """Inverses of the principal submatrices of the level operator on each cell's nodes and all time nodes."""
        n, dim = self.k + 1, self.dim
        zero = self.mus.index((0,) * self.spec["M"])
        Ml = torch.einsum("q,qa,qb->ab", self.w, self.phi, self.phi)
        Kl = sum(torch.einsum("cq,qa,qb->cab", self.a[zero] * self.w, g, g) for g in self.grad)
        shape = list(reversed(self.cells))
        Kl = Kl.reshape(shape + [n ** dim, n ** dim])
        Mp, Kp = torch.zeros_like(Kl), torch.zeros_like(Kl)
        local = np.stack([g.reshape(-1) for g in reversed(np.meshgrid(*[np.arange(n)] * dim, indexing="ij"))])
        for off in np.ndindex(*[3] * dim):
            o = np.array(off) - 1                                                # neighbour cell + o, x first
            other = local - self.k * o[:, None]
            ok = np.all((other >= 0) & (other <= self.k), axis=0)
            here = torch.as_tensor(np.flatnonzero(ok), device="cuda")
            there = torch.as_tensor((other[:, ok] * (n ** np.arange(dim))[:, None]).sum(0), device="cuda")
            to = tuple(slice(max(0, -o[d]), self.cells[d] - max(0, o[d])) for d in reversed(range(dim)))
            fr = tuple(slice(max(0, o[d]), self.cells[d] - max(0, -o[d])) for d in reversed(range(dim)))
            Kp[to + (here[:, None], here[None])] += Kl[fr + (there[:, None], there[None])]
            Mp[to + (here[:, None], here[None])] += Ml[there[:, None], there[None]]
        Mp, Kp = Mp.flatten(0, dim - 1), Kp.flatten(0, dim - 1)
        m = self.inner[self.conn]
        m2 = (m[:, :, None] * m[:, None, :])[:, None, :, None, :]
        A = (self.At[:, None, :, None] * Mp[:, None, :, None, :] + self.Bt[:, None, :, None] * Kp[:, None, :, None, :]) * m2
        A = A.reshape(A.shape[0], self.nt * n ** dim, -1)
        A += torch.diag_embed((1 - m).repeat(1, self.nt))
        inv = torch.linalg.inv(A)
        return inv.float().bfloat16().double() if factors == "bf16" else inv


def _triples(rows, mu, cols):
    """E[Psi_a Psi_mu Psi_b] by Gauss-Hermite quadrature in each variable."""
    n = max(max(map(max, rows)), max(map(max, cols))) + 1
    y, w = np.polynomial.hermite_e.hermegauss(2 * n + max(mu) + 1)
    w = w / w.sum()
    v = np.array([_psi(i, y) for i in range(n)])
    out = np.ones((len(rows), len(cols)))
    for m, d in enumerate(mu):
        t = np.einsum("q,iq,jq->ij", w * _psi(d, y), v, v)
        t[np.abs(t) < 1e-12] = 0.0
        out *= t[np.ix_([a[m] for a in rows], [b[m] for b in cols])]
    return out


class _Forcing:
    """Load vectors of the manufactured solution: f = u_t - div(a grad u), tested with (k+4)-point Gauss rules."""

    def __init__(self, case, spec, samples=None):
        self.P, man = _Plain(spec, n_gauss=spec["k"] + 4, samples=samples), _manufactured(case)
        P, M = self.P, spec["M"]
        idx_q = _indices(M, man["q"])
        self.T = np.poly1d(man["T"][::-1])
        arg = [np.pi / (spec["hi"][d] - spec["lo"][d]) for d in range(P.dim)]
        val, der = [], []
        for c, f in zip(man["c"], man["freq"]):
            s = [np.sin(arg[d] * f[d] * (P.x[d] - spec["lo"][d])) for d in range(P.dim)]
            co = [arg[d] * f[d] * np.cos(arg[d] * f[d] * (P.x[d] - spec["lo"][d])) for d in range(P.dim)]
            val.append(c * math.prod(s))
            der.append([c * math.prod(co[e] if e == d else s[e] for e in range(P.dim)) for d in range(P.dim)])
        val, der = _t(np.array(val)), _t(np.array(der))
        if samples is not None:
            psi = _t(np.array([[np.prod([_psi(a, x) for a, x in zip(al, xi)]) for al in idx_q] for xi in samples]))
            val, grad = torch.einsum("sa,acq->scq", psi, val), torch.einsum("sa,adcq->dscq", psi, der)
            flux = [P.couple(g[:, None])[:, 0] for g in grad]
        else:
            idx = _indices(M, spec["P"])
            flux = [sum(a * torch.einsum("ba,acq->bcq", _t(_triples(idx, mu, idx_q)), der[:, d]) for mu, a in zip(P.mus, P.a))
                    for d in range(P.dim)]
            pick = _t(np.array([[float(a == b) for a in idx_q] for b in idx]))
            val = torch.einsum("ba,acq->bcq", pick, val)
        once = lambda f, t: P.scatter(((f * P.w) @ t)[:, None])[:, 0]  # noqa: E731
        self.mass, self.stiff = once(val, P.phi), sum(once(f, g) for f, g in zip(flux, P.grad))

    def load(self, slab):
        P = self.P
        x, w = _gauss(P.nt + 4)
        v = _lagrange(P.t_nodes, x)[0]
        t = P.tau * (slab + x)
        a, b = (_t(P.tau * (w * f(t)) @ v)[None, :, None] for f in (self.T.deriv(), self.T))
        F = a * self.mass[:, None] + b * self.stiff[:, None]
        return F + _t(P.v0)[None, :, None] * float(self.T(0.0)) * self.mass[:, None] if slab == 0 else F


def _previous(c, seed):
    """The state of a march before slab 1: the manufactured solution's nodal values, a little disturbed."""
    spec, man = _spec(c, seed), _manufactured(c)
    tau = spec["T"] / spec["n_slabs"]
    idx, idx_q = _indices(c["M"], c["P"]), _indices(c["M"], 2)
    node, pos = _lobatto(c["k"]), []
    for d in range(c["dim"]):
        n = _cells(c)[d]
        x = np.concatenate([(i + node[:-1]) / n for i in range(n)] + [[1.0]])
        pos.append(x)
    u = np.zeros((len(idx), c["r"] + 1, math.prod(len(x) for x in pos)))
    for a, cc, f in zip(idx_q, man["c"], man["freq"]):
        if a in idx:
            s = np.sin(np.pi * f[0] * pos[0])
            for d in range(1, c["dim"]):
                s = np.multiply.outer(np.sin(np.pi * f[d] * pos[d]), s)
            for i, t in enumerate(tau * _radau(c["r"])):
                u[idx.index(a), i] = cc * (t + t * t) * s.reshape(-1)
    return _t(u.reshape(-1)) + 1e-3 * tau * _random(c, seed, True)


def exact(case, seed):
    c = case
    spec, kind = _spec(c, seed), c["kind"]
    if kind == "apply":
        return _Plain(spec).apply(_random(c, seed, False), c.get("trans", False)).reshape(-1)
    if kind == "vcycle":
        return _Plain(spec, diagonal=True).vcycle(_random(c, seed, True), c["mg"], 0.9).reshape(-1)
    if kind == "solve":
        return _Plain(spec).solve(_random(c, seed, True)).reshape(-1)
    if kind == "march":
        P = _Plain(spec)
        rhs = _Forcing(c, spec).load(1) + P.mass(_previous(c, seed), P.Ct)
        u = P.solve(rhs)
        return {"rhs": rhs.reshape(-1), "y": u.reshape(-1), "mean": u[0, -1].clone(), "var": u[1:, -1].square().sum(0)}
    if kind == "mc":
        xi = _samples(c, seed)
        P, F, u = _Plain(spec, samples=xi), _Forcing(c, spec, xi), None
        for n in range(c["slabs"]):
            u = P.solve(F.load(n) + (P.mass(u, P.Ct) if n else 0.0))
        return {"mean": u[:, -1].mean(0), "var": u[:, -1].var(0, unbiased=True), "paths": u.reshape(-1)}
    P, F, us = _Plain(spec), _Forcing(c, spec), []
    for n in range(c["slabs"]):
        us.append(P.solve(F.load(n) + (P.mass(us[-1], P.Ct) if n else 0.0)))
    last = torch.zeros_like(P.At)
    last[-1, -1] = 1.0
    mu = P.mass(us[-1], last)
    J, src = float((us[-1] * mu).sum()), 2 * mu
    amp, cell = np.zeros(len(P.pieces)), 0.0
    for u in reversed(us):
        lam = P.solve(src, trans=True)
        src = P.mass(lam, P.Ct.T.contiguous())
        gu, gl = P.gather(u), P.gather(lam)
        # per term: lam . (G B) grad u at every point; weighted by each piece's own field
        for t, (mu_t, G) in enumerate(zip(P.mus, P.G)):
            dens = sum(((G.T @ (gl @ g.T).flatten(1)).view(-1, P.nt, *P.a[0].shape) *
                        torch.einsum("ij,ajcq->aicq", P.Bt, gu @ g.T)).sum((0, 1)) for g in P.grad) * P.w
            for i, p in enumerate(P.pieces):
                if tuple(p["mu"]) == mu_t:
                    amp[i] -= float((dens * _t(P.field(p))).sum())
                    if i == 0:
                        cell = cell - p["amp"] * (dens * _t(P.field(p, scaled=False))).sum(1)
    return {"J": J, "amp": amp, "cell": cell.cpu().numpy()}
