"""The tuner against a plan's own choices: the value that a plan has is tried and
kept where it is the fastest, whether or not it is among the listed ones, and a
cached entry serves only the kernels, grid class and top boundary that it was
tuned on."""
import json

import pytest

from paper_2103_01874_gb300 import autotune, ppe

# launch shapes with a time of 10 us at the plan's own choice and more elsewhere
KERNELS = {"rhs_lines": "k_rhs_march", "rhs_planes": "k_rhs_march", "x_lines": "k_xinv", "z_cols": "k_zfft_fwd",
           "y_cols": "k_ysolve"}


class Plan:
    nx, ny, nz, precision = 64, 64, 64, 1

    def __init__(self, bc_top=ppe.BC_WALL, **own):
        self.opts = ppe.Options(ppe.FP32_REFINE, 0, 1e-10, 4, 1e-12, bc_top)
        self.own = dict(dict(rhs_lines=2, rhs_planes=8, x_lines=16, z_cols=16, y_cols=8, spectral=0, y_solve=0), **own)
        self.t, self.rec, self.on = dict(self.own), {}, False

    def get_tuning(self):
        return dict(self.t)

    def set_tuning(self, **kw):
        if kw.get("spectral", 0) or kw.get("y_solve", 0):
            raise ppe.PPEError(1, "ppe_set_tuning")
        self.t.update(kw)

    def profile(self, on):
        self.on = on

    def profile_read(self):
        rec, self.rec = self.rec, {}
        return rec

    def run(self, k):
        if self.on:
            for name in set(KERNELS.values()):
                us = 10 + sum(abs(self.t[f] - self.own[f]) for f, kn in KERNELS.items() if kn == name)
                self.rec[name] = (k, 1e-3 * us * k)


@pytest.mark.parametrize("field,value", [("rhs_planes", n) for n in (1, 2, 3, 5, 6, 7, 10, 12)]
                         + [("rhs_lines", 2), ("x_lines", 2), ("z_cols", 1), ("y_cols", 1)])
def test_own_choice_is_kept_where_it_is_the_fastest(field, value, tmp_path):
    plan = Plan(**{field: value})
    res = autotune.autotune(plan, plan.run, reps=1, path=str(tmp_path / "t.json"))
    assert res["tuning"] == plan.own == plan.get_tuning()


def test_cached_entry_serves_its_own_class_only(tmp_path, monkeypatch):
    path = str(tmp_path / "t.json")
    tuned = Plan(rhs_planes=2)
    autotune.autotune(tuned, tuned.run, reps=1, path=path, search={"rhs_planes": autotune.SEARCH["rhs_planes"]})
    same, other = Plan(), Plan(bc_top=ppe.BC_OUTFLOW)
    assert autotune.apply_cached(same, path) and same.get_tuning()["rhs_planes"] == 2
    assert not autotune.apply_cached(other, path) and other.get_tuning() == other.own
    # an entry of a key without the sources, as earlier builds wrote it, or of other sources
    doc = json.load(open(path))
    (entry,) = doc.values()
    gpu = autotune._gpu_name()
    json.dump({f"64x64x64|prec1|face0|{gpu}": entry}, open(path, "w"))
    assert not autotune.apply_cached(Plan(), path)
    autotune.save_cache(doc, path)
    monkeypatch.setattr(autotune, "kernels_version", lambda: "other")
    assert not autotune.apply_cached(Plan(), path)
