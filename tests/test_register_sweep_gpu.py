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


def _bytes_per_cell(by_cell):
    """Device bytes per finest cell of a one-row Q2 dG(1) hierarchy whose patch
    inverses take `by_cell`: with them three FP32 vectors (4 nodes, 2 time
    nodes), two FP64 coefficient tables of 9 points and one in FP32, and a
    third as much again for the coarser levels."""
    return 4.0 / 3.0 * (by_cell + 3 * 4 * 2 * 4 + 2 * 9 * 8 + 9 * 4)


@pytest.mark.parametrize("prec,value", [(sg.SG_PREC_FP32, 4), (sg.SG_PREC_BF16, 2)], ids=["fp32", "bf16"])
def test_inverses_are_held_once(cuda, prec, value):
    """Set-up takes no more memory than with the inverses by cell alone (18
    rows of 24 values), 16 MB aside for what does not grow with the mesh."""
    ctx = sg.sg_setup_spec(_spec((512, 512), 2, 1, 1, 0))
    sg.sg_mg_setup(ctx, prec)                       # loads the kernels
    warm = sg.sg_setup_spec(_spec((512, 512), 2, 1, 1, 0))
    cuda.cuda.synchronize()
    before = cuda.cuda.mem_get_info()[0]
    sg.sg_mg_setup(warm, prec)
    assert sg.sg_mg_level_info(warm, 0)["vanka_kind"] == 2
    taken = before - cuda.cuda.mem_get_info()[0]
    ctx.destroy()
    warm.destroy()
    assert taken <= 512 * 512 * _bytes_per_cell(18 * 24 * value) + (16 << 20), taken / 512 ** 2


@pytest.mark.parametrize("prec", [sg.SG_PREC_FP32, sg.SG_PREC_BF16], ids=["fp32", "bf16"])
@pytest.mark.parametrize("k,r,cells", [(2, 1, (10, 14)), (1, 3, (36, 4))])
def test_inverses_in_either_order(cuda, k, r, cells, prec):
    """A forced variant puts the inverses back by cell: the same values."""
    ctx = sg.sg_setup_spec(_spec(cells, k, r, 2, 2))
    sg.sg_mg_set_coarse_dofs(ctx, 0)
    sg.sg_mg_setup(ctx, prec)
    last = cells[0] * cells[1] - 1
    where = [(0, 0), (0, 5), (0, 31), (0, 32), (0, last)] + ([(1, last // 4)] if sg.sg_mg_level_info(ctx, 0)["levels"] > 2 else [])
    first = [sg.sg_mg_patch_inverse(ctx, lev, 0, c) for lev, c in where]
    sg.sg_mg_set_level_variant(ctx, -1, -1, 1, 0, 0)
    assert sg.sg_mg_level_info(ctx, 0)["vanka_kind"] == 0
    for a, (lev, c) in zip(first, where):
        assert np.array_equal(a, sg.sg_mg_patch_inverse(ctx, lev, 0, c))
    ctx.destroy()


def test_no_room_for_both_orders(cuda):
    """With room for the inverses by cell but not for both orders at once,
    set-up succeeds with another sweep (1024^2 cells: 2.8 GB in all, the finest
    level's inverses alone 3.4 GB in both orders) and the V-cycle agrees to FP32."""
    spec, n = _spec((1024, 1024), 2, 1, 1, 0), 1024 * 1024
    ctx = sg.sg_setup_spec(spec)
    sg.sg_mg_setup(ctx, sg.SG_PREC_FP32)
    assert sg.sg_mg_level_info(ctx, 0)["vanka_kind"] == 2
    r = cuda.from_numpy(np.random.default_rng(4).uniform(-1, 1, ctx.info["n_unknowns"])).cuda()
    want, got = cuda.empty_like(r), cuda.full_like(r, float("nan"))
    sg.sg_vcycle(ctx, r, want)
    sg.sg_mg_set_level_variant(ctx, -1, -1, 2, 0, 0)      # loads the other sweep
    sg.sg_vcycle(ctx, r, got)
    ctx.destroy()
    ctx = sg.sg_setup_spec(spec)
    cuda.cuda.synchronize()
    cuda.cuda.empty_cache()
    hold = cuda.empty(cuda.cuda.mem_get_info()[0] - 2900 * n, dtype=cuda.uint8, device="cuda")
    try:
        sg.sg_mg_setup(ctx, sg.SG_PREC_FP32)
        assert sg.sg_mg_level_info(ctx, 0)["vanka_kind"] == 0
        got.fill_(float("nan"))
        sg.sg_vcycle(ctx, r, got)
        err = float((got - want).abs().max() / want.abs().max())
    finally:
        del hold
        cuda.cuda.empty_cache()
    ctx.destroy()
    assert err < 1e-4, err
