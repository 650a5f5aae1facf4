"""Double-word apply over the range of its two floats: scaling the input by a
power of two scales every exact result by it, so the apply of the scaled vector
must match the oracle's apply to the same 1e-12 as the unscaled one (the
rounding of a double-word sum to one double works on its exponent and bits)."""
import numpy as np
import pytest

import paper_2605_21046_gb300 as sg
from oracle import operator
from paper_2605_21046_gb300 import inputs as I

pytestmark = pytest.mark.gpu

CASES = {
    "2d-q2-13x7": dict(I.config_small_2d_q1(), cells=(13, 7), k=2),
    "3d-q1-5x4x3": I.scaled(dict(I.config_3d_q2_32(), k=1), (5, 4, 3)),
}


@pytest.mark.parametrize("log2", [-60, -1, 0, 40, 90])
@pytest.mark.parametrize("name", list(CASES))
def test_scaled_input(cuda, name, log2):
    spec = CASES[name]
    x = I.random_vector(spec, seed=6)
    want = operator.SGProblem(spec).apply(x).reshape(-1)
    ctx = sg.sg_setup_spec(spec, sg.SG_PREC_DW)
    xd = cuda.from_numpy(np.ldexp(x, log2)).cuda()
    yd = cuda.full_like(xd, float("nan"))
    sg.sg_apply(ctx, 0, xd, yd)
    got = np.ldexp(yd.cpu().numpy(), -log2)
    ctx.destroy()
    err = float(np.abs(got - want).max() / np.abs(want).max())
    assert err < 1e-12, err
