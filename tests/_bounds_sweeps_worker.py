"""Worker of the second debug-bounds GPU test: run in a fresh process with
SG_DEBUG_BOUNDS=1.  The kernels that set-up picks by itself, before any variant
is forced: register sweeps in both directions at partial warps, transfers in
tiles of columns, the device's coarse inverse and the coarse solve; prints one
JSON line with the records."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def main():
    import torch
    import paper_2605_21046_gb300 as sg
    from paper_2605_21046_gb300 import _abi
    from paper_2605_21046_gb300 import inputs as I

    def spec(cells, k, r, M=3, P=2, coef=None):
        dim = len(cells)
        freqs = [tuple(((m + d) % 3) + 1 for d in range(dim)) for m in range(M)]
        return dict(name="bounds", dim=dim, cells=cells, lo=(0.0,) * dim, hi=(1.0,) * dim, k=k, r=r, n_slabs=3, T=1.0, M=M,
                    P=P, coef=coef or I.linear_sine_coef(M, dim, 0.08, freqs))

    out = {"library": os.path.basename(_abi.load()._name)}
    sg.sg_debug_bounds()                                      # clear
    # 10 modes: the last block of 4 rows is partly empty; the squared coefficient: several classes
    sweeps = [spec((10, 14), 2, 1), spec((36, 4), 2, 0), spec((6, 22), 1, 3), spec((12, 20), 1, 2),
              spec((8, 6), 2, 1, 4, 2, I.paper_coefficient())]
    for s in sweeps:
        for prec in (sg.SG_PREC_FP32, sg.SG_PREC_BF16):
            ctx = sg.sg_setup_spec(s)
            sg.sg_mg_set_coarse_dofs(ctx, 0)
            sg.sg_mg_setup(ctx, prec)
            assert sg.sg_mg_level_info(ctx, 0)["vanka_kind"] == 2
            n = ctx.info["n_unknowns"]
            b = torch.rand(n, dtype=torch.float64, device="cuda")
            sg.sg_vcycle(ctx, b, torch.empty_like(b))
            sg.sg_solve_slab_adjoint(ctx, 0, b, torch.zeros_like(b), rtol=1e-6)
            sg.sg_mg_set_level_variant(ctx, -1, -1, 1, 0, 0)  # the inverses back by cell
            sg.sg_vcycle(ctx, b, torch.empty_like(b))
            ctx.destroy()
    out["after_sweeps"] = sg.sg_debug_bounds()
    for cells, k, prec in (((1384, 16), 2, sg.SG_PREC_FP64), ((608, 16), 3, sg.SG_PREC_FP64), ((2848, 32), 2, sg.SG_PREC_BF16)):
        ctx = sg.sg_setup_spec(spec(cells, k, 0, 1, 0))
        sg.sg_mg_setup(ctx, prec)
        b = torch.rand(ctx.info["n_unknowns"], dtype=torch.float64, device="cuda")
        sg.sg_vcycle(ctx, b, torch.empty_like(b))
        ctx.destroy()
    out["after_long_rows"] = sg.sg_debug_bounds()
    # coarse operators around the blocks of 16 pivots and tiles of 32
    for s in (spec((3, 2), 1, 0), spec((5, 5), 1, 0), spec((4, 4), 1, 1), spec((12, 4), 1, 0), spec((5, 3), 2, 1),
              spec((3, 3, 3), 2, 1)):
        for prec in (sg.SG_PREC_FP64, sg.SG_PREC_FP32):
            ctx = sg.sg_setup_spec(s)
            sg.sg_mg_setup(ctx, prec)
            b = torch.rand(ctx.info["n_unknowns"], dtype=torch.float64, device="cuda")
            sg.sg_vcycle(ctx, b, torch.empty_like(b))
            sg.sg_solve_slab_adjoint(ctx, 0, b, torch.zeros_like(b), rtol=1e-6)
            ctx.destroy()
    out["after_coarse"] = sg.sg_debug_bounds()
    print(json.dumps(out), flush=True)


if __name__ == "__main__":
    main()
