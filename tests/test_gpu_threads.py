"""Plans that launch the same kernel instances with different amounts of dynamic
shared memory, in turn and from two host threads with a stream each: the
right-hand side at nx = 128 (two stacks of lines per CTA at ny = 128, three at
96) and the x passes of a length without an instance at two tiles.  Every call
succeeds and gives the bits of the plan alone."""
import threading

import pytest

from _gpu_util import dev_fields
from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu

PAIRS = [(((128, 128, 8), {}), ((128, 96, 8), {}), ppe.FP32_REFINE),
         (((108, 16, 12), {"x_lines": 32}), ((108, 16, 12), {"x_lines": 64}), ppe.FP64)]


@pytest.mark.parametrize("a,b,prec", PAIRS)
def test_two_sizes_of_one_instance(a, b, prec):
    import torch
    jobs = []
    for n, (shape, tune) in enumerate((a, b)):
        fl = fields.make_fields(*shape, seed=41 + n, recipe="single", width=3.0)
        st = torch.cuda.Stream()
        plan = ppe.Plan(*shape, fl.lx, fl.ly, fl.lz, precision=prec, stream=st)
        plan.set_tuning(**tune)
        jobs.append(dict(plan=plan, d=dev_fields(fl), dt=fl.dt, st=st))
    torch.cuda.synchronize()

    def outs(j):
        return [torch.zeros_like(j["d"][k]) for k in ("rho", "u", "v", "w")]

    def project(j, o):
        d = j["d"]
        j["plan"].project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], j["dt"], *o)

    for j in jobs:
        j["want"] = outs(j)
    torch.cuda.synchronize()
    for j in jobs:
        project(j, j["want"])
    torch.cuda.synchronize()
    for j in jobs:  # in turn: the smaller size after the larger and before it
        j["got"] = outs(j)
    torch.cuda.synchronize()
    for _ in range(3):
        for j in jobs:
            project(j, j["got"])
    torch.cuda.synchronize()
    for j in jobs:
        assert all(torch.equal(x, y) for x, y in zip(j["want"], j["got"]))
        j["got"] = outs(j)
    torch.cuda.synchronize()
    errors = []

    def loop(j):
        try:
            for _ in range(300):
                project(j, j["got"])
        except Exception as e:  # noqa: BLE001 - reported below
            errors.append(e)

    threads = [threading.Thread(target=loop, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for j in jobs:
        assert all(torch.equal(x, y) for x, y in zip(j["want"], j["got"]))
        j["plan"].close()
