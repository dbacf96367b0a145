"""Fields of very small magnitude, down to below what the float pairs hold
(2^-126): the linear problem scaled by s gives s times the result up to the
pairs' absolute resolution, and is neither reported as incompatible nor as not
converged.

Bounds, with Kc = rho_0/dt and h the spacings: a pair's absolute error below 2^-126
is at most 2^-126, so f differs by at most Kc 2^-126 (2/hx + 2/hy + 2/hz + 1), p by
that times half the squared box (the maximum principle), a velocity by 2^-126 plus
(dt/rho_0) 2/h times p's; and 1e-8 relative for the scaled result (the refinement's
1e-10 and the condition number of this grid)."""
import numpy as np
import pytest

from _gpu_util import dev_fields, to_dev
from oracle import ppe_oracle as O
from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu

SHAPE = (32, 24, 32)
SCALES = [1e-10, 1e-18, 1e-20, 1e-22, 1e-24, 1e-28, 1e-31, 1e-33, 1e-34, 1e-35, 1e-36, 1e-37, 1e-38, 1e-39, 1e-40,
          1e-44, 1e-100, 1e-300]
TINY = 2.0 ** -126


def _fields():
    return fields.make_fields(*SHAPE, seed=3, recipe="multimode", width=3.0, rho_g=60.0)


def _outs(d):
    import torch
    return {k: torch.zeros_like(d[s]) for k, s in (("p", "rho"), ("u", "u"), ("v", "v"), ("w", "w"))}


@pytest.mark.parametrize("prec", [ppe.FP32_REFINE, ppe.FP64])
@pytest.mark.parametrize("top", [ppe.BC_WALL, ppe.BC_OUTFLOW])
def test_projection_of_scaled_fields(prec, top):
    fl = _fields()
    ref = O.project_fields(fl, bc_top=top)
    d0 = dev_fields(fl)
    h = O.spacings(fl.shape, (fl.lx, fl.ly, fl.lz))
    kc = fl.rho.min() / fl.dt
    p_abs = kc * TINY * (sum(2 / x for x in h) + 1) * (fl.lx ** 2 + fl.ly ** 2 + fl.lz ** 2) / 2
    v_abs = TINY + 2 / min(h) / kc * p_abs
    with ppe.Plan(*SHAPE, fl.lx, fl.ly, fl.lz, precision=prec, bc_top=top) as plan:
        for s in SCALES:
            d = {k: (t if k == "rho" else t * s) for k, t in d0.items()}
            o = _outs(d)
            plan.project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], fl.dt, *o.values())
            plan.info()  # neither incompatible nor unconverged
            for k in o:
                e = np.abs(o[k].cpu().numpy() - s * ref[k]).max()
                assert e <= 1e-8 * s * np.abs(ref[k]).max() + (p_abs if k == "p" else v_abs), (s, k, e)


@pytest.mark.parametrize("prec", [ppe.FP32_REFINE, ppe.FP64])
def test_solve_of_a_scaled_right_hand_side(prec):
    import torch
    fl = _fields()
    f = np.random.default_rng(5).normal(size=fl.shape)
    f -= f.mean()
    ref = O.ppe_solve(f, (fl.lx, fl.ly, fl.lz))
    p_abs = TINY * (fl.lx ** 2 + fl.ly ** 2 + fl.lz ** 2) / 2
    with ppe.Plan(*SHAPE, fl.lx, fl.ly, fl.lz, precision=prec) as plan:
        for s in SCALES:
            p = torch.zeros(fl.shape, dtype=torch.float64, device="cuda")
            plan.solve(to_dev(s * f), p)
            plan.info()
            e = np.abs(p.cpu().numpy() - s * ref).max()
            assert e <= 1e-8 * s * np.abs(ref).max() + p_abs, (s, e)


def test_incompatible_small_fields_are_still_reported():
    fl = _fields()
    d0 = dev_fields(fl)
    with ppe.Plan(*SHAPE, fl.lx, fl.ly, fl.lz) as plan:
        for s in (1.0, 1e-10, 1e-20, 1e-25):
            d = {k: (t if k == "rho" else t * s) for k, t in d0.items()}
            o = _outs(d)
            plan.project(d["u"], d["v"], d["w"], d["S"] + 1e-3 * s, d["rho"], d["p_n"], d["p_nm1"], fl.dt, *o.values())
            with pytest.raises(ppe.PPEError) as e:
                plan.info()
            assert e.value.code == 3


@pytest.mark.parametrize("prec", [ppe.FP32_REFINE, ppe.FP64])
def test_unsplit_of_vanishing_fields(prec):
    """Below 2^-74 the unsplit projection takes g for zero and keeps the velocities."""
    fl = _fields()
    d0 = dev_fields(fl)
    with ppe.Plan(*SHAPE, fl.lx, fl.ly, fl.lz, precision=prec) as plan:
        for s in (1e-24, 1e-28, 1e-33, 1e-36, 1e-38, 1e-40, 1e-44, 1e-100, 1e-300):
            d = {k: (t if k == "rho" else t * s) for k, t in d0.items()}
            o = _outs(d)
            plan.project_unsplit(d["u"], d["v"], d["w"], d["S"], d["rho"], fl.dt, *o.values())
            plan.unsplit_info()
            assert float(o["p"].abs().max()) == 0.0
            for k in ("u", "v", "w"):
                assert float((o[k] - d[k]).abs().max()) <= TINY + 2.0 ** -46 * s * float(d0[k].abs().max())
