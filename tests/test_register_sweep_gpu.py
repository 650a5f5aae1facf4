"""The register Vanka sweep (FP32 vectors, 2D patches of at most 18 unknowns),
which set-up picks by itself on such levels."""
import numpy as np
import pytest

import paper_2605_21046_gb300 as sg
from paper_2605_21046_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _spec(cells, k, r, M, P, hi=(1.0, 1.0), coef=None):
    freqs = [((m % 3) + 1, ((m + 1) % 3) + 1) for m in range(M)]
    return dict(name="reg", dim=2, cells=cells, lo=(0.0, 0.0), hi=hi, k=k, r=r, n_slabs=4, T=1.0, M=M, P=P,
                coef=coef or I.linear_sine_coef(M, 2, 0.08, freqs))


@pytest.mark.parametrize("prec", [sg.SG_PREC_FP32, sg.SG_PREC_BF16], ids=["fp32", "bf16"])
def test_more_cells_than_a_grid_axis_of_tiles(cuda, prec):
    """2048 x 1024 cells: 65536 tiles of 32 cells.  The same V-cycle with the
    shared-memory sweep, which stores the inverses by cell (FP32: 1e-4)."""
    ctx = sg.sg_setup_spec(_spec((2048, 1024), 1, 0, 1, 0, hi=(2.0, 1.0)))
    sg.sg_mg_setup(ctx, prec)
    assert sg.sg_mg_level_info(ctx, 0)["vanka_kind"] == 2
    r = cuda.from_numpy(np.random.default_rng(4).uniform(-1, 1, ctx.info["n_unknowns"])).cuda()
    got, want = cuda.full_like(r, float("nan")), cuda.full_like(r, float("nan"))
    sg.sg_vcycle(ctx, r, got)
    sg.sg_mg_set_level_variant(ctx, -1, -1, 2, 0, 0)
    sg.sg_vcycle(ctx, r, want)
    err = float((got - want).abs().max() / want.abs().max())
    ctx.destroy()
    assert err < 1e-4, err
