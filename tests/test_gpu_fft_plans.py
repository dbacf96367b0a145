"""The register-staged FP32 passes at every length with a split plan (a factor
3, or 16 and 32 points), in each direction, at the smallest and largest tiles,
with walls and an open top, against the numpy oracle: residual <= 1e-10 (the
refinement's target), f <= 1e-12, u, v, w <= 1e-11 as for the other lengths
(<= 1e-8 with the open top, whose one-sweep result is held to its residual).
These grids are thin, so p's lowest modes magnify the residual by the grid's
condition number (up to 2e5 at 384 cells): p is held to the residual and,
through its gradient, to the velocities."""
import numpy as np
import pytest

from _gpu_util import dev_fields
from oracle import ppe_oracle as O
from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu

SHAPES = [(2 * n, 9, 8) for n in (16, 24, 32, 48, 96, 192)] + [(18, n, 9) for n in (16, 24, 32, 48, 96, 192, 384)] + \
         [(12, 8, n) for n in (16, 24, 32, 48, 96, 192, 384)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("top", [ppe.BC_WALL, ppe.BC_OUTFLOW])
def test_split_plan_lengths(shape, top):
    import torch
    nx, ny, nz = shape
    h = 2.0 * np.pi / ny
    fl = fields.make_fields(nx, ny, nz, seed=nx + ny + nz, recipe="multimode", width=3.0, rho_g=60.0, lx=0.9 * h * nx,
                            lz=1.1 * h * nz)
    ref = O.project_fields(fl, bc_top=top)
    d = dev_fields(fl)
    o = {k: torch.empty_like(d[s]) for k, s in (("p", "rho"), ("u", "u"), ("v", "v"), ("w", "w"), ("f", "rho"))}
    with ppe.Plan(nx, ny, nz, fl.lx, fl.ly, fl.lz, precision=ppe.FP32_REFINE, bc_top=top) as plan:
        for tiles in (dict(), dict(x_lines=1, z_cols=1, y_cols=1), dict(x_lines=64, z_cols=16, y_cols=32)):
            plan.set_tuning(**tiles)
            plan.project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], fl.dt, o["p"], o["u"], o["v"],
                         o["w"], f=o["f"])
            assert plan.info().rel_residual <= 1e-10
            f, p = o["f"].cpu().numpy(), o["p"].cpu().numpy()
            assert O.rel_linf(f, ref["f"]) <= 1e-12
            r = O.residual(f, p, (fl.lx, fl.ly, fl.lz), bc_top=top)
            assert np.abs(r - (r.mean() if top == ppe.BC_WALL else 0.0)).max() <= 1e-10 * np.abs(f).max()
            for k in ("u", "v", "w"):
                assert O.rel_linf(o[k].cpu().numpy(), ref[k]) <= (1e-11 if top == ppe.BC_WALL else 1e-8), k
