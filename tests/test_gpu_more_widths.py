"""Widths between those that the other files run: the x passes of 384 points
(nx = 768, the three-pass split plan) with walls and an open top, to the bounds of
the other split plans (residual 1e-10, f 1e-12, u, v, w 1e-11 with walls and 1e-8
with the open top, p through its residual); and every height of the right-hand
side's column stacks at the widths with an instance of their own (the bits of the
default height)."""
import numpy as np
import pytest

from _gpu_util import dev_fields
from oracle import ppe_oracle as O
from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("top", [ppe.BC_WALL, ppe.BC_OUTFLOW])
def test_x_passes_of_384_points(top):
    import torch
    nx, ny, nz = 768, 9, 8
    h = 2.0 * np.pi / ny
    fl = fields.make_fields(nx, ny, nz, seed=7, recipe="multimode", width=3.0, rho_g=60.0, lx=0.9 * h * nx,
                            lz=1.1 * h * nz)
    ref = O.project_fields(fl, bc_top=top)
    d = dev_fields(fl)
    o = {k: torch.empty_like(d[s]) for k, s in (("p", "rho"), ("u", "u"), ("v", "v"), ("w", "w"), ("f", "rho"))}
    with ppe.Plan(nx, ny, nz, fl.lx, fl.ly, fl.lz, precision=ppe.FP32_REFINE, bc_top=top) as plan:
        for x_lines in (4, 1, 64):
            try:
                plan.set_tuning(x_lines=x_lines)
            except ppe.PPEError:
                continue  # (64 lines of 768 cells do not fit)
            plan.project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], fl.dt, o["p"], o["u"], o["v"],
                         o["w"], f=o["f"])
            assert plan.info().rel_residual <= 1e-10
            f, p = o["f"].cpu().numpy(), o["p"].cpu().numpy()
            assert O.rel_linf(f, ref["f"]) <= 1e-12
            r = O.residual(f, p, (fl.lx, fl.ly, fl.lz), bc_top=top)
            assert np.abs(r - (r.mean() if top == ppe.BC_WALL else 0.0)).max() <= 1e-10 * np.abs(f).max()
            for k in ("u", "v", "w"):
                assert O.rel_linf(o[k].cpu().numpy(), ref[k]) <= (1e-11 if top == ppe.BC_WALL else 1e-8), k


@pytest.mark.parametrize("nx", [32, 64, 96, 128, 192, 256])
@pytest.mark.parametrize("rule,rho0", [(ppe.FACE_ARITHMETIC, -1.0), (ppe.FACE_HARMONIC, 55.0)])
def test_heights_of_the_compiled_widths(nx, rule, rho0):
    import torch
    fl = fields.make_fields(nx, 54, 9, seed=nx, recipe="multimode", width=4.0, rho_g=60.0)
    d = dev_fields(fl)
    want = None
    with ppe.Plan(nx, 54, 9, fl.lx, fl.ly, fl.lz, face_rule=rule) as plan:
        for lines in (2, 1, 4, 8):
            for planes in (4, 1, 9):
                plan.set_tuning(rhs_lines=lines, rhs_planes=planes)
                o = [torch.zeros_like(d[k]) for k in ("rho", "u", "v", "w", "rho")]
                plan.project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], fl.dt, *o[:4], f=o[4],
                             rho0=rho0)
                torch.cuda.synchronize()
                got = [t.cpu().numpy() for t in o]
                want = want or got
                for a, b in zip(want, got):
                    assert np.array_equal(a, b), (lines, planes)
