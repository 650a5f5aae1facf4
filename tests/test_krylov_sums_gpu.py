"""FGMRES with short bases: the reductions of the Gram-Schmidt passes take up to
2, 4, 8 or 16 sums at once, and groups of 16 beyond that.  A restart of 2, 3, 5,
9 and 17 runs every count up to it, one count past each boundary."""
import numpy as np
import pytest

import paper_2605_21046_gb300 as sg
from paper_2605_21046_gb300 import inputs as I
from oracle import operator, solver

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("restart,omega", [(2, 0.5), (3, 0.5), (5, 0.3), (9, 0.2), (17, 0.1)])
def test_restarted_solves_match_the_oracle(cuda, restart, omega):
    """Iterations within one of the oracle's FGMRES with the same V-cycle and
    restart; the true residual at most 1.5 x the tolerance (the solver tests' bound)."""
    torch = cuda
    spec = I.config_small_2d_q1()
    p = operator.SGProblem(spec)
    b = np.random.default_rng(7).uniform(-1, 1, p.shape)
    b[:, :, p.bmask] = 0.0
    _, its, _ = solver.fgmres(p, b, solver.Multigrid(p, nu=1, omega=omega, coarse_dofs=0).apply, rtol=1e-10,
                              restart=restart)
    assert its > restart
    ctx = sg.sg_setup_spec(spec)
    sg.sg_mg_set_coarse_dofs(ctx, 0)
    sg.sg_mg_setup(ctx, sg.SG_PREC_FP64, 1, omega)
    x = torch.zeros(b.size, dtype=torch.float64, device="cuda")
    st = sg.sg_solve_slab(ctx, 0, torch.from_numpy(b.reshape(-1).copy()).cuda(), x, rtol=1e-10, max_it=300,
                          restart=restart)
    got = x.cpu().numpy()
    ctx.destroy()
    res = np.linalg.norm(b.reshape(-1) - p.apply(got).reshape(-1)) / np.linalg.norm(b)
    assert st["converged"] == 1 and res <= 1.5e-10, (res, st)
    assert abs(st["iterations"] - its) <= 1, (st["iterations"], its)
