"""z planes per right-hand-side CTA in the graph form of a batch: a plan's own
choice is raised to min(8, nz), a value that a call gave is taken as it is, also
where it equals the plan's own choice, and ppe_get_tuning reports it unchanged.
The wall flux (one partial sum per wall tile and chunk of planes) shows by its
bits which chunks ran."""
import numpy as np
import pytest

from _gpu_util import to_dev
from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu

SEEDS = range(6)


@pytest.mark.parametrize("shape", [(64, 48, 32), (96, 64, 32)])
def test_given_planes_are_kept_in_a_batch(shape):
    import torch

    def plan_and_fields(seed):
        fl = fields.make_fields(*shape, seed=seed, recipe="single", width=3.0)
        d = {k: to_dev(v) for k, v in fl.arrays().items()}
        walls = np.random.default_rng(seed).normal(size=(shape[2], 2, shape[0]))
        d["v"][:, 0], d["v"][:, -1] = to_dev(walls[:, 0]), to_dev(walls[:, 1])
        d.update(p=torch.empty_like(d["rho"]), u_out=torch.empty_like(d["u"]), v_out=torch.empty_like(d["v"]),
                 w_out=torch.empty_like(d["w"]), dt=fl.dt)
        return ppe.Plan(*shape, fl.lx, fl.ly, fl.lz, precision=ppe.FP32_REFINE), d

    def flux(pl):
        return pl.info(allow_not_converged=True, allow_incompatible=True).wall_flux_mean

    def direct(planes):
        out = []
        for s in SEEDS:
            pl, d = plan_and_fields(s)
            pl.set_tuning(rhs_planes=planes)
            pl.project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], d["dt"], d["p"], d["u_out"],
                       d["v_out"], d["w_out"])
            out.append(flux(pl))
            pl.close()
        return out

    def batch(prepare):
        items = [plan_and_fields(s) for s in SEEDS]
        for pl, _ in items:
            before = pl.get_tuning()
            prepare(pl, before["rhs_planes"])
            assert pl.get_tuning() == before
        with ppe.Batch(items, form=ppe.BATCH_GRAPH) as b:
            b.launch()
            torch.cuda.synchronize()
        out = [flux(pl) for pl, _ in items]
        for pl, _ in items:
            pl.close()
        return out

    def refused(pl, own):
        with pytest.raises(ppe.PPEError):
            pl.set_tuning(rhs_planes=own, rhs_lines=3)

    def given_then_refused(pl, own):
        pl.set_tuning(rhs_planes=own)
        refused(pl, own)

    own = plan_and_fields(0)[0].get_tuning()["rhs_planes"]
    assert own < 8
    at_own, at_eight = direct(own), direct(8)
    assert at_own != at_eight  # (the sums' grouping shows)
    assert np.allclose(at_own, at_eight, rtol=1e-12, atol=0)
    assert batch(lambda pl, own: None) == at_eight
    assert batch(lambda pl, own: pl.set_tuning(y_cols=pl.get_tuning()["y_cols"])) == at_eight
    assert batch(refused) == at_eight
    assert batch(lambda pl, own: pl.set_tuning(rhs_planes=own)) == at_own
    assert batch(given_then_refused) == at_own
