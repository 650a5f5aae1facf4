"""A hierarchy of one level: the V-cycle is the dense solve of every diagonal
block, so it must equal the oracle's exact block solve (Sec. 3.5 remark).
Sizes around the device elimination's blocks of 16 pivots and tiles of 32, and
an indefinite block (negative mean coefficient), where its unpivoted
elimination may fail its check and the pivoting one takes over.  FP64, 1e-10
as for the other V-cycle comparisons."""
import numpy as np
import pytest

import paper_2605_21046_gb300 as sg
from oracle import operator, solver
from paper_2605_21046_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _spec(cells, k, r, a0=1.0):
    dim = len(cells)
    return dict(name="coarse", dim=dim, cells=cells, lo=(0.0,) * dim, hi=(1.0,) * dim, k=k, r=r, n_slabs=4, T=1.0, M=2, P=1,
                coef=I.linear_sine_coef(2, dim, 0.05, [(1,) * dim, (2,) * dim], a0=a0))


CASES = {
    "2": _spec((3, 2), 1, 0),
    "16": _spec((5, 5), 1, 0),
    "18": _spec((4, 4), 1, 1),
    "33": _spec((12, 4), 1, 0),
    "90": _spec((5, 3), 2, 1),
    "250-3d": _spec((3, 3, 3), 2, 1),
    "507": _spec((7, 7), 2, 2),
    "indefinite": _spec((5, 4), 2, 1, a0=-1.0),
}


@pytest.mark.parametrize("trans", [False, True], ids=["forward", "transposed"])
@pytest.mark.parametrize("name", list(CASES))
def test_one_level_is_the_exact_block_solve(cuda, name, trans):
    spec = CASES[name]
    p = operator.SGProblem(spec)
    b = np.random.default_rng(8).uniform(-1, 1, p.shape)
    b[:, :, np.asarray(p.bmask)] = 0.0
    mg = solver.Multigrid(p)
    assert len(mg.levels) == 1
    ctx = sg.sg_setup_spec(spec)
    sg.sg_mg_setup(ctx, sg.SG_PREC_FP64)
    assert sg.sg_mg_level_info(ctx, 0)["levels"] == 1
    bd = cuda.from_numpy(b.reshape(-1).copy()).cuda()
    if not trans:
        zd = cuda.full_like(bd, float("nan"))
        sg.sg_vcycle(ctx, bd, zd)
        want, got = mg.apply(b).reshape(-1), zd.cpu().numpy()
        err = float(np.abs(got - want).max() / np.abs(want).max())
        assert err < 1e-10, err
    else:
        # the transposed cycle preconditions the adjoint solve
        xd = cuda.zeros_like(bd)
        sg.sg_solve_slab_adjoint(ctx, 0, bd, xd, rtol=1e-12, max_it=60)
        res = p.apply(xd.cpu().numpy(), transpose=True).reshape(-1) - b.reshape(-1)
        assert np.linalg.norm(res) <= 1e-10 * np.linalg.norm(b)
    ctx.destroy()
