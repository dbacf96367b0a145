"""ppe_rhs at the widths with an instance of their own, on tiles that end past the
top wall and with one-plane chunks: the bits of the f that the projection forms,
and within 1e-12 of the numpy oracle (the bound of f elsewhere)."""
import numpy as np
import pytest

from _gpu_util import dev_fields
from oracle import ppe_oracle as O
from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(32, 36, 9), (64, 27, 8), (96, 9, 16), (128, 18, 8), (192, 9, 12), (256, 27, 8),
                                   (384, 9, 8), (48, 27, 9), (512, 8, 9)])
@pytest.mark.parametrize("rule", [ppe.FACE_ARITHMETIC, ppe.FACE_HARMONIC])
@pytest.mark.parametrize("rho0", [-1.0, 2500.0])
@pytest.mark.parametrize("top", [ppe.BC_WALL, ppe.BC_OUTFLOW])
def test_rhs_alone(shape, rule, rho0, top):
    import torch
    nx, ny, nz = shape
    h = 2.0 * np.pi / ny
    fl = fields.make_fields(nx, ny, nz, seed=nx + ny, recipe="single", width=3.0, lx=0.8 * h * nx, lz=1.3 * h * nz)
    ref = O.project_fields(fl, rule=rule, rho0=rho0 if rho0 > 0 else None, bc_top=top)["f"]
    d = dev_fields(fl)
    with ppe.Plan(nx, ny, nz, fl.lx, fl.ly, fl.lz, face_rule=rule, bc_top=top) as plan:
        for planes in (plan.get_tuning()["rhs_planes"], 1, nz):
            plan.set_tuning(rhs_planes=planes)
            o = [torch.zeros_like(d[k]) for k in ("rho", "u", "v", "w", "rho")]
            plan.project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], fl.dt, *o[:4], f=o[4],
                         rho0=rho0)
            f = torch.zeros_like(d["rho"])
            plan.rhs(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], fl.dt, f, rho0=rho0)
            assert torch.equal(f, o[4])
            assert O.rel_linf(f.cpu().numpy(), ref) <= 1e-12
