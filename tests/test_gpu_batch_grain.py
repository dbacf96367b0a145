"""The persistent batch's item size: radix-3 z and y passes take several
consecutive tiles of an item at once, whatever the number of tiles left and
where the plane ends, so every grain (one tile per item, odd runs, long runs)
gives the same bits."""
import numpy as np
import pytest

from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu

# 48, 96 and 192 points in y and z; 3, 5, 7, 9 and 13 tiles of 8 columns, 2, 3, 5 and 7 of 16, per line of tiles
SHAPES = [(32, 48, 96), (64, 96, 48), (96, 192, 192), (128, 48, 48), (192, 96, 96), (48, 192, 64)]


def test_grain_changes_no_bit():
    import torch
    items = []
    for n, shape in enumerate(SHAPES):
        fl = fields.make_fields(*shape, seed=60 + n, recipe="single", width=2.0)
        d = {k: torch.from_numpy(v.copy()).to("cuda") for k, v in fl.arrays().items()}
        d.update(p=torch.empty_like(d["rho"]), u_out=torch.empty_like(d["u"]), v_out=torch.empty_like(d["v"]),
                 w_out=torch.empty_like(d["w"]), dt=fl.dt)
        items.append((ppe.Plan(*shape, fl.lx, fl.ly, fl.lz, precision=ppe.FP32_REFINE), d))
    ref = None
    for grain in (1, 2000, 16384, 100000):
        with ppe.Batch(items, form=ppe.BATCH_PERSISTENT, grain=grain) as b:
            b.launch()
            assert b.status()["status"] == 0
        got = [d[k].cpu().numpy() for _, d in items for k in ("p", "u_out", "v_out", "w_out")]
        assert all(np.isfinite(g).all() for g in got)
        ref = ref or got
        assert all(np.array_equal(a, c) for a, c in zip(ref, got)), grain
    for pl, _ in items:
        assert pl.info().rel_residual <= 1e-10
        pl.close()
