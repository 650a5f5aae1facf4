"""One reduction of a double-word value h + l into a double where h is a power of
two and l points towards zero: a last place below h is half as large there.
Inputs scaled so that a chosen result is 2^k (1 - 2^-27).  At a cell's centre
(Q2) it comes from one cell, in one reduction.  A wrong step would be off by
2^-27 of it; the bound is 1e-12 of the largest interior result, as for the
unscaled applies."""
import numpy as np
import pytest

import paper_2605_21046_gb300 as sg
from oracle import operator
from paper_2605_21046_gb300 import inputs as I

pytestmark = pytest.mark.gpu
SPEC = dict(I.config_small_2d_q1(), cells=(13, 7), k=2)


def _apply(torch, x):
    ctx = sg.sg_setup_spec(SPEC, sg.SG_PREC_DW)
    xd = torch.from_numpy(x).cuda()
    yd = torch.full_like(xd, float("nan"))
    sg.sg_apply(ctx, 0, xd, yd)
    y = yd.cpu().numpy()
    ctx.destroy()
    return y


def _interior():
    return np.tile(~I.boundary_mask(SPEC), I.n_modes(SPEC) * (SPEC["r"] + 1))


@pytest.mark.parametrize("sign", [1, -1])
def test_results_just_inside_a_power_of_two(cuda, sign):
    x = I.random_vector(SPEC, seed=7)
    want = operator.SGProblem(SPEC).apply(x).reshape(-1)
    nx, ny = (2 * c + 1 for c in SPEC["cells"])
    node = np.arange(nx * ny)
    centre = np.tile((node % nx % 2 == 1) & (node // nx % 2 == 1), want.size // node.size)
    top = np.abs(want[_interior()]).max()
    chosen = np.flatnonzero(centre & (np.abs(want) >= 0.3 * top) & (np.sign(want) == sign))[:6]
    assert chosen.size == 6
    for i in chosen:
        k = np.floor(np.log2(abs(want[i])))
        s = 2.0 ** k * (1 - 2.0 ** -27) / abs(want[i])
        got = _apply(cuda, s * x)[i]
        assert abs(got - s * want[i]) <= 1e-12 * top, (i, got - s * want[i])
