"""The dense coarse solve of indefinite operators (a negative mean coefficient):
an elimination in order can lose digits there without failing, so its inverse
must be refused and the pivoting one taken.  One-level hierarchies, where the
V-cycle is the coarse solve X b of every mode.

Bound: with the oracle's operator C and inverse, |C (X b) - b| relative to the
largest entry of |C| |C^-1| |b|, in units of 2^-52.  The library accepts an
inverse at 8 on one vector; 64 leaves a factor of 8 for another vector.  The
elimination in order is at 438, 2406 and 4968 on these three (its arithmetic
repeated in numpy), a pivoting one below 1."""
import numpy as np
import pytest

import paper_2605_21046_gb300 as sg
from oracle import operator, solver
from paper_2605_21046_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = {"q3-dg3-5x5-0.05": ((5, 5), 3, 3, -0.05), "q3-dg3-5x5-0.01": ((5, 5), 3, 3, -0.01), "q2-dg1-5x4": ((5, 4), 2, 1, -0.01)}


@pytest.mark.parametrize("name", list(CASES))
def test_indefinite_coarse_solve_keeps_its_digits(cuda, name):
    cells, k, r, a0 = CASES[name]
    spec = dict(name="coarse", dim=2, cells=cells, lo=(0.0, 0.0), hi=(1.0, 1.0), k=k, r=r, n_slabs=4, T=1.0, M=2, P=1,
                coef=I.linear_sine_coef(2, 2, 0.05, [(1, 1), (2, 2)], a0=a0))
    p = operator.SGProblem(spec)
    b = np.random.default_rng(8).uniform(-1, 1, p.shape)
    b[:, :, np.asarray(p.bmask)] = 0.0
    ctx = sg.sg_setup_spec(spec)
    sg.sg_mg_setup(ctx, sg.SG_PREC_FP64)
    assert sg.sg_mg_level_info(ctx, 0)["levels"] == 1
    bd = cuda.from_numpy(b.reshape(-1).copy()).cuda()
    zd = cuda.full_like(bd, float("nan"))
    sg.sg_vcycle(ctx, bd, zd)
    z = zd.cpu().numpy().reshape(b.shape[0], -1)
    ctx.destroy()
    mg = solver.Multigrid(p)
    L = mg.levels[0]
    for a in range(b.shape[0]):
        C = L.A[mg.cls[a]][L.inner][:, L.inner].toarray()
        rhs = b[a].reshape(-1)[L.inner]
        off = np.abs(C @ z[a][L.inner] - rhs).max()
        size = (np.abs(C) @ (np.abs(L.Ainv[mg.cls[a]]) @ np.abs(rhs))).max()
        assert off <= 64 * 2.0 ** -52 * size, off / size * 2.0 ** 52


@pytest.mark.parametrize("prec", [sg.SG_PREC_FP64, sg.SG_PREC_FP32, sg.SG_PREC_BF16], ids=["fp64", "fp32", "bf16"])
def test_set_up_without_interior_nodes(cuda, prec):
    """A row of Q1 cells has boundary nodes only: set-up has nothing to invert,
    and the operator is the identity."""
    spec = dict(name="row", dim=2, cells=(4, 1), lo=(0.0, 0.0), hi=(1.0, 1.0), k=1, r=1, n_slabs=4, T=1.0, M=1, P=1,
                coef=I.linear_sine_coef(1, 2, 0.1, [(1, 1)]))
    ctx = sg.sg_setup_spec(spec)
    sg.sg_mg_setup(ctx, prec)
    assert sg.sg_mg_level_info(ctx, 0)["coarsest"] == 1
    x = cuda.from_numpy(I.random_vector(spec)).cuda()
    y = cuda.full_like(x, float("nan"))
    sg.sg_apply(ctx, 0, x, y)
    assert cuda.equal(x, y)
    ctx.destroy()
