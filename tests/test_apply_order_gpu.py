"""An apply right behind a kernel that writes its input, and right before one
that overwrites it, on the same stream: the cell kernel starts while the pass
that presets y still runs, and must not be ahead of anything else.  Against the
same applies with the device idle around each (two FP64 runs differ by the order
of their reductions: 1e-13 of the largest result; double-word 1e-12)."""
import pytest

import paper_2605_21046_gb300 as sg
from paper_2605_21046_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SPECS = {
    "8x8": I.config_small_2d_q1(),
    "45x37": dict(I.scaled(I.config_2d_q2_64(), (45, 37)), P=2),
    "3d-12": I.scaled(I.config_3d_q2_32(), (12, 12, 12)),
}


@pytest.mark.parametrize("side", [False, True], ids=["default", "side-stream"])
@pytest.mark.parametrize("prec", [sg.SG_PREC_FP64, sg.SG_PREC_DW], ids=["fp64", "dw"])
@pytest.mark.parametrize("name", list(SPECS))
def test_apply_between_writers_of_its_input(cuda, name, prec, side):
    torch, spec = cuda, SPECS[name]
    ctx = sg.sg_setup_spec(spec, prec)
    n = ctx.info["n_unknowns"]
    g = torch.Generator(device="cuda").manual_seed(3)
    src = [torch.rand(n, generator=g, dtype=torch.float64, device="cuda") - 0.5 for _ in range(4)]
    want = []
    for s in src:
        y = torch.empty_like(s)
        torch.cuda.synchronize()
        sg.sg_apply(ctx, 0, s, y)
        torch.cuda.synchronize()
        want.append(y)
    x = torch.empty(n, dtype=torch.float64, device="cuda")
    out = [torch.full_like(x, float("nan")) for _ in range(40)]
    torch.cuda.synchronize()
    st = torch.cuda.Stream() if side else torch.cuda.current_stream()
    with torch.cuda.stream(st):
        for i, y in enumerate(out):
            x.copy_(src[i % 4])
            sg.sg_apply(ctx, 0, x, y)
            x.fill_(float("nan"))
    torch.cuda.synchronize()
    ctx.destroy()
    tol = 1e-13 if prec == sg.SG_PREC_FP64 else 1e-12
    for i, y in enumerate(out):
        w = want[i % 4]
        assert float((y - w).abs().max()) <= tol * float(w.abs().max()), i
