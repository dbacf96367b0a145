"""Right-hand side on grids 258 to 512 wide at every accepted height of its column
stacks (one, two or four lines, with ragged last tiles and chunks of planes),
both face rules: the projection's outputs have the bits of the default shape
and ppe_rhs is within 1e-12 of the numpy oracle (the bound of the default shape
elsewhere); a height whose tile would be too large is refused."""
import numpy as np
import pytest

from _gpu_util import dev_fields
from oracle import ppe_oracle as O
from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(288, 27, 9), (324, 16, 8), (384, 9, 8), (486, 12, 9), (512, 27, 9)])
@pytest.mark.parametrize("rule", [ppe.FACE_ARITHMETIC, ppe.FACE_HARMONIC])
def test_stack_heights_of_wide_grids(shape, rule):
    import torch
    nx, ny, nz = shape
    h = 2.0 * np.pi / ny
    fl = fields.make_fields(nx, ny, nz, seed=nx + ny, recipe="single", width=3.0, lx=0.8 * h * nx, lz=1.3 * h * nz)
    ref = O.project_fields(fl, rule=rule)
    d = dev_fields(fl)
    with ppe.Plan(nx, ny, nz, fl.lx, fl.ly, fl.lz, face_rule=rule) as plan:

        def project():
            o = [torch.zeros_like(d[k]) for k in ("rho", "u", "v", "w", "rho")]
            plan.project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], fl.dt, *o[:4], f=o[4])
            torch.cuda.synchronize()
            return [t.cpu().numpy() for t in o]

        default = project()
        assert O.rel_linf(default[4], ref["f"]) <= 1e-12
        heights = [n for n in (1, 2, 4, 8) if n * nx <= 2048]
        for lines, planes in [(n, k) for n in heights for k in (1, 5, nz)]:
            plan.set_tuning(rhs_lines=lines, rhs_planes=planes)
            for a, b in zip(default, project()):
                assert np.array_equal(a, b), (lines, planes)
            f = torch.zeros_like(d["rho"])
            plan.rhs(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], fl.dt, f)
            assert O.rel_linf(f.cpu().numpy(), ref["f"]) <= 1e-12, (lines, planes)
        for lines in {1, 2, 4, 8} - set(heights):
            with pytest.raises(ppe.PPEError):
                plan.set_tuning(rhs_lines=lines)
