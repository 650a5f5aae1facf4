"""Grid transfers of levels whose rows are too long for one block's shared
memory: tiles of columns (the first counts of cells along x that need them, and
one that no tile divides).  The V-cycle commutes with exchanging the axes, and
with x and y (z) exchanged the rows are short, so the V-cycle of the exchanged
problem must be the exchanged V-cycle: FP64 1e-10, FP32 1e-4, as for the other
V-cycle comparisons.  One case against the oracle as well."""
import numpy as np
import pytest

import paper_2605_21046_gb300 as sg
from oracle import operator, solver
from paper_2605_21046_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _spec(cells, k, freqs, hi):
    dim = len(cells)
    return dict(name="long", dim=dim, cells=cells, lo=(0.0,) * dim, hi=hi, k=k, r=0, n_slabs=4, T=1.0, M=1, P=1,
                coef=I.linear_sine_coef(1, dim, 0.3, [freqs]))


def _vcycle(torch, spec, prec, r):
    """V-cycle of r (rows, nodes in the spec's axis order, x last)."""
    ctx = sg.sg_setup_spec(spec)
    sg.sg_mg_setup(ctx, prec)
    rd = torch.from_numpy(np.ascontiguousarray(r).reshape(-1)).cuda()
    zd = torch.full_like(rd, float("nan"))
    sg.sg_vcycle(ctx, rd, zd)
    got = zd.cpu().numpy().reshape(r.shape)
    ctx.destroy()
    return got


CASES = {
    "q1-fp64": ((6464, 16), 1, sg.SG_PREC_FP64),
    "q2-fp64": ((1384, 16), 2, sg.SG_PREC_FP64),
    "q3-fp64": ((608, 16), 3, sg.SG_PREC_FP64),
    "q1-fp32": ((12928, 16), 1, sg.SG_PREC_FP32),
    "q2-bf16": ((2848, 32), 2, sg.SG_PREC_BF16),
    "q3-fp32": ((1216, 32), 3, sg.SG_PREC_FP32),
    "3d-q2-fp64": ((1408, 32, 32), 2, sg.SG_PREC_FP64),
}


@pytest.mark.parametrize("name", list(CASES))
def test_long_rows_match_the_exchanged_problem(cuda, name):
    cells, k, prec = CASES[name]
    dim = len(cells)
    freqs, hi = (3,) + (1, 2)[:dim - 1], (cells[0] / cells[1],) + (1.0, 0.7)[:dim - 1]     # nearly square cells
    shape = (2,) + tuple(k * c + 1 for c in reversed(cells))
    r = np.random.default_rng(12).uniform(-1, 1, shape)
    got = _vcycle(cuda, _spec(cells, k, freqs, hi), prec, r)
    swap = lambda a: a.swapaxes(1, dim)  # noqa: E731
    want = swap(_vcycle(cuda, _spec(cells[::-1], k, freqs[::-1], hi[::-1]), prec, swap(r)))
    err = float(np.abs(got - want).max() / np.abs(want).max())
    assert err < (1e-10 if prec == sg.SG_PREC_FP64 else 1e-4), err


def test_long_rows_match_the_oracle(cuda):
    cells, k, prec = CASES["q3-fp64"]
    spec = _spec(cells, k, (3, 1), (cells[0] / cells[1], 1.0))
    p = operator.SGProblem(spec)
    r = np.random.default_rng(13).uniform(-1, 1, p.shape)
    want = solver.Multigrid(p).apply(r).reshape(r.shape)
    got = _vcycle(cuda, spec, prec, r)
    err = float(np.abs(got - want).max() / np.abs(want).max())
    assert err < 1e-10, err
