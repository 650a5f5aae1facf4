"""V-cycles on meshes whose rows of cells do not fill a warp and whose chaos
rows do not fill a block, against the oracle: odd and rectangular levels,
anisotropic cells, several diagonal classes, every time degree (Sec. 3.5
remark; the level residual by the row-diagonal apply, FP64 1e-10, FP32 1e-4 as
for the other V-cycle comparisons)."""
import numpy as np
import pytest

import paper_2605_21046_gb300 as sg
from oracle import operator, solver
from paper_2605_21046_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _spec(cells, k, r, M, P, hi, coef=None):
    dim = len(cells)
    freqs = [tuple(((m + d) % 3) + 1 for d in range(dim)) for m in range(M)]
    return dict(name="edge", dim=dim, cells=cells, lo=(-0.5,) * dim, hi=hi, k=k, r=r, n_slabs=4, T=1.0, M=M, P=P,
                coef=coef or I.linear_sine_coef(M, dim, 0.08, freqs))


CASES = {
    "2d-q2-20x12-dg1": _spec((20, 12), 2, 1, 2, 2, (1.0, 0.7)),           # 6 rows, 33-node lines over two warps
    "2d-q2-36x4-dg0": _spec((36, 4), 2, 0, 2, 2, (1.0, 1.0)),             # a row longer than a warp
    "2d-q2-512x8-dg0": _spec((512, 8), 2, 0, 1, 0, (1.0, 1.0)),           # transfer rows beyond 48 KB of shared memory
    "2d-q1-12x20-dg2": _spec((12, 20), 1, 2, 3, 1, (0.4, 1.0)),
    "2d-q3-8x6-dg3-classes": _spec((8, 6), 3, 3, 4, 2, (0.5, 0.5), I.paper_coefficient()),
    "3d-q2-6x4x8": _spec((6, 4, 8), 2, 1, 2, 1, (1.0, 0.5, 0.8)),
    "3d-q1-10x6x4-dg0": _spec((10, 6, 4), 1, 0, 1, 2, (1.0, 1.0, 0.5)),
}


@pytest.mark.parametrize("prec,tol", [(sg.SG_PREC_FP64, 1e-10), (sg.SG_PREC_FP32, 1e-4)], ids=["fp64", "fp32"])
@pytest.mark.parametrize("name", list(CASES))
def test_vcycle_matches_oracle(cuda, name, prec, tol):
    spec = CASES[name]
    p = operator.SGProblem(spec)
    r = np.random.default_rng(5).uniform(-1, 1, p.shape)
    want = solver.Multigrid(p, coarse_dofs=0).apply(r).reshape(-1)
    ctx = sg.sg_setup_spec(spec)
    sg.sg_mg_set_coarse_dofs(ctx, 0)
    sg.sg_mg_setup(ctx, prec)
    sg.sg_mg_set_level_variant(ctx, -1, 1)
    rd = cuda.from_numpy(r.reshape(-1).copy()).cuda()
    zd = cuda.full_like(rd, float("nan"))
    sg.sg_vcycle(ctx, rd, zd)
    got = zd.cpu().numpy()
    ctx.destroy()
    err = float(np.abs(got - want).max() / np.abs(want).max())
    assert err < tol, err
