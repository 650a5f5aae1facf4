"""Writes sg_shape_tables.h: the reference-cell tables of Q_k (k = 1..3) on
[0, 1] as compile-time constants, so that the compiler folds their exact zeros
and ones out of the sum-factorisation passes.

  S[q][n]  = l_n(g_q): Gauss-Lobatto Lagrange basis l_n at the (k+1) Gauss points g_q
  D[q][p]  = L_p'(g_q): derivative of the Lagrange basis L_p on the Gauss points
  L[i]     = the constants of the 1D passes of Q2 and Q3 (Line in sg_apply_kernel.cuh), in
             the order of its enumerators, and W, the square of the unit its derivatives
             are taken in; each rounded once (derived from S and D in double they cost Q3
             half as much error again)
  Sh/Sl, Dh/Dl: the same values as float pairs hi + lo (hi = value rounded to
  float, lo = the remainder rounded to float), for double-word arithmetic

Values are computed with 40-digit arithmetic and rounded once to double.
sg_setup recomputes both tables in double precision and refuses to run if
they differ by more than 1e-13 (a guard against a stale header).

    python gen_shape_tables.py   # rewrites sg_shape_tables.h beside this file
"""
import os

import mpmath as mp
import numpy as np

mp.mp.dps = 40


def gauss(n):
    xs = [(mp.mpf(1) + x) / 2 for x in sorted(mp.polyroots(mp.taylor(lambda t: mp.legendre(n, t), 0, n)[::-1], maxsteps=200, extraprec=200))]
    return xs


def lobatto(k):
    if k == 1:
        return [mp.mpf(0), mp.mpf(1)]
    if k == 2:
        return [mp.mpf(0), mp.mpf(1) / 2, mp.mpf(1)]
    s = 1 / mp.sqrt(5)
    return [mp.mpf(0), (1 - s) / 2, (1 + s) / 2, mp.mpf(1)]


def lag(nodes, i, t):
    v = mp.mpf(1)
    for j, xj in enumerate(nodes):
        if j != i:
            v *= (t - xj) / (nodes[i] - xj)
    return v


def dlag(nodes, i, t):
    s = mp.mpf(0)
    for k, xk in enumerate(nodes):
        if k == i:
            continue
        term = 1 / (nodes[i] - xk)
        for j, xj in enumerate(nodes):
            if j != i and j != k:
                term *= (t - xj) / (nodes[i] - xj)
        s += term
    return s


def lit(v):
    v = float(v)
    if abs(v) < 1e-30:
        return "0.0"
    return repr(v)


def split(v):
    h = np.float32(float(v))
    lo = np.float32(float(v - mp.mpf(float(h))))
    return h, lo


def flit(f):
    f = np.float32(f)
    if f == 0:
        return "0.0f"
    return repr(float(f)) + "f"


def table(name, n, vals, typ, fmt):
    body = ", ".join("{" + ", ".join(fmt(vals[a][b]) for b in range(n)) + "}" for a in range(n))
    return [f"  __host__ __device__ static constexpr {typ} {name}(int a, int b) {{",
            f"    constexpr {typ} t[{n}][{n}] = {{{body}}};",
            "    return t[a][b];", "  }"]


def line_constants(k, S, D):
    """(constants, squared derivative unit) of the 1D passes."""
    if k == 1:
        return [mp.mpf(0)], mp.mpf(1)
    if k == 2:
        return [mp.mpf(3) / 10, mp.mpf(4) / 10, (S[2][2] - S[2][0]) / 2, mp.mpf(12) / 10], D[1][2] ** 2
    unit = (D[3][3] - D[3][0]) / 2
    even = lambda T, q, n: (T[q][n] + T[q][3 - n]) / 2  # noqa: E731
    odd = lambda T, q, n: (T[q][n] - T[q][3 - n]) / 2  # noqa: E731
    co, ci, co1, ci0 = odd(S, 3, 3), odd(S, 2, 2), odd(S, 3, 2), odd(S, 2, 3)
    qo, qi = even(D, 3, 3) / unit, even(D, 2, 3) / unit
    ai, bo, bi = odd(D, 2, 3) / unit, odd(D, 3, 2) / unit, odd(D, 2, 2) / unit
    return [even(S, 3, 3), even(S, 3, 2), even(S, 2, 3), even(S, 2, 2), co, ci, co1 / co, ci0 / ci, ci0 / co, co1 / ci,
            ai, bo, bi, qo, qi, 2 * qo, 2 * qi, 2 * ai, 2 * bo, 2 * bi], unit ** 2


def main():
    out = ["// Generated by gen_shape_tables.py - do not edit.",
           "// Reference Q_k tables on [0,1] at the (k+1)-point Gauss rule.",
           "#pragma once", "", "namespace sg {", "",
           "template <int K> struct RefShape;", ""]
    for k in (1, 2, 3):
        g = gauss(k + 1)
        nodes = lobatto(k)
        n = k + 1
        S = [[lag(nodes, j, g[q]) for j in range(n)] for q in range(n)]
        D = [[dlag(g, p, g[q]) for p in range(n)] for q in range(n)]
        # exact zeros / ones stay exact
        def clean(v):
            if abs(v) < mp.mpf(10) ** -30:
                return mp.mpf(0)
            if abs(v - 1) < mp.mpf(10) ** -30:
                return mp.mpf(1)
            return v
        S = [[clean(v) for v in row] for row in S]
        D = [[clean(v) for v in row] for row in D]
        Sh = [[split(v)[0] for v in row] for row in S]
        Sl = [[split(v)[1] for v in row] for row in S]
        Dh = [[split(v)[0] for v in row] for row in D]
        Dl = [[split(v)[1] for v in row] for row in D]
        out.append(f"template <> struct RefShape<{k}> {{")
        out.append(f"  static constexpr int N = {n};")
        out += table("S", n, S, "double", lit)
        out += table("D", n, D, "double", lit)
        out += table("Sh", n, Sh, "float", flit)
        out += table("Sl", n, Sl, "float", flit)
        out += table("Dh", n, Dh, "float", flit)
        out += table("Dl", n, Dl, "float", flit)
        L, W = line_constants(k, S, D)
        out += [f"  static constexpr double W = {lit(W)};",
                "  __host__ __device__ static constexpr double L(int i) {",
                f"    constexpr double t[{len(L)}] = {{{', '.join(lit(v) for v in L)}}};",
                "    return t[i];", "  }"]
        out.append("};")
        out.append("")
    out.append("}  // namespace sg")
    path = os.path.join(os.path.dirname(os.path.abspath(__file__)), "sg_shape_tables.h")
    open(path, "w").write("\n".join(out) + "\n")
    print(path)


if __name__ == "__main__":
    main()
