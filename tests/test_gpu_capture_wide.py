"""A caller's capture of projections whose kernels take more than 48 KB of shared
memory: right-hand-side tiles of 87 KB (128 x 96), 95 KB (384 wide) and the x
passes of a length without an instance, with the plan's first call inside the
capture.  Replays give the bits of direct calls."""
import pytest

from _gpu_util import dev_fields
from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,tune", [((128, 96, 16), {}), ((384, 9, 8), {}), ((108, 16, 12), {"x_lines": 64}),
                                        ((192, 24, 9), {"rhs_lines": 8})])
@pytest.mark.parametrize("prec", [ppe.FP32_REFINE, ppe.FP64])
def test_capture_of_large_tiles(shape, tune, prec):
    import torch
    fl = fields.make_fields(*shape, seed=5, recipe="single", width=3.0)
    d = dev_fields(fl)
    st = torch.cuda.Stream()
    with ppe.Plan(*shape, fl.lx, fl.ly, fl.lz, precision=prec, stream=st) as plan:
        plan.set_tuning(**tune)

        def project(o):
            plan.project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], fl.dt, *o)

        got, want = ([torch.zeros_like(d[k]) for k in ("rho", "u", "v", "w")] for _ in range(2))
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            project(got)
        for _ in range(2):
            for t in got:
                t.zero_()
            torch.cuda.synchronize()
            graph.replay()
            torch.cuda.synchronize()
        with torch.cuda.stream(st):
            project(want)
        torch.cuda.synchronize()
        assert all(float(t.abs().max()) > 0 for t in got)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
        plan.info()
