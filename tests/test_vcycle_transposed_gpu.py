"""The transposed V-cycle element by element.  It has no entry point of its own,
but the first FGMRES iterate of the transposed solve from zero is z scaled by
the minimiser of |b - c A^T z|, z = P^-T b:  x = c z, c = <A^T z, b> / |A^T z|^2.

The oracle's V-cycle with every level operator, patch inverse and coarse
inverse transposed gives z (bf16 factors: rounded, then transposed).  FP64
1e-10, FP32 vectors 1e-4, as for the forward V-cycles.  The forward V-cycle's
iterate is checked to differ, so that a sweep that forgot to transpose fails."""
import numpy as np
import pytest

import paper_2605_21046_gb300 as sg
from oracle import operator, solver
from paper_2605_21046_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _spec(cells, k, r, M=3, P=1, coef=None):
    dim = len(cells)
    freqs = [tuple(((m + d) % 3) + 1 for d in range(dim)) for m in range(M)]
    return dict(name="trans", dim=dim, cells=cells, lo=(0.0,) * dim, hi=(1.0, 0.8, 0.9)[:dim], k=k, r=r, n_slabs=2, T=1.0,
                M=M, P=P, coef=coef or I.linear_sine_coef(M, dim, 0.08, freqs))


CASES = {
    "2d-q2-dg1": (_spec((10, 12), 2, 1), 2),
    "2d-q1-dg3": (_spec((36, 4), 1, 3), 2),
    "2d-q1-dg2-classes": (_spec((6, 12), 1, 2, 4, 2, I.paper_coefficient()), 2),
    "2d-q2-dg2": (_spec((8, 6), 2, 2), None),
    "2d-q3-dg1": (_spec((4, 8), 3, 1), None),
    "3d-q2-dg1": (_spec((4, 4, 6), 2, 1, 1, 1), None),
}
PREC = {"fp64": (sg.SG_PREC_FP64, 1e-10), "fp32": (sg.SG_PREC_FP32, 1e-4), "bf16": (sg.SG_PREC_BF16, 1e-4)}


def _transpose(mg):
    for L in mg.levels:
        L.A = [a.T.tocsr() for a in L.A]
        if L.coarsest:
            L.Ainv = [m.T for m in L.Ainv]
        else:
            L.patch_inv = [[m.T for m in inv] for inv in L.patch_inv]


def _first_iterate(p, z, b):
    w = p.apply(z, transpose=True).reshape(-1)
    return (w @ b.reshape(-1)) / (w @ w) * z.reshape(-1)


@pytest.mark.parametrize("prec", list(PREC))
@pytest.mark.parametrize("name", list(CASES))
def test_transposed_vcycle_matches_oracle(cuda, name, prec):
    spec, register = CASES[name]
    p = operator.SGProblem(spec)
    b = np.random.default_rng(14).uniform(-1, 1, p.shape)
    mg = solver.Multigrid(p, factor_round=solver.round_bf16 if prec == "bf16" else None, coarse_dofs=0)
    forward = _first_iterate(p, mg.apply(b), b)
    _transpose(mg)
    want = _first_iterate(p, mg.apply(b), b)
    code, tol = PREC[prec]
    ctx = sg.sg_setup_spec(spec)
    sg.sg_mg_set_coarse_dofs(ctx, 0)
    sg.sg_mg_setup(ctx, code)
    assert len(mg.levels) >= 2 and sg.sg_mg_level_info(ctx, 0)["levels"] == len(mg.levels)
    if register and prec != "fp64":
        assert sg.sg_mg_level_info(ctx, 0)["vanka_kind"] == register
    x = cuda.zeros(b.size, dtype=cuda.float64, device="cuda")
    st = sg.sg_solve_slab_adjoint(ctx, 0, cuda.from_numpy(b.reshape(-1).copy()).cuda(), x, rtol=1e-14, max_it=1, check=False)
    got = x.cpu().numpy()
    ctx.destroy()
    assert st["iterations"] == 1
    scale = np.abs(want).max()
    err = float(np.abs(got - want).max() / scale)
    assert err < tol, err
    assert np.abs(forward - want).max() > 1e-3 * scale
