"""A caller's own capture of projections: on a stream joined from another one
(the first kernel has two predecessors, one of them a copy), several calls of
both precisions in a row, with walls and an open top.  Replays give the bits of
direct calls."""
import numpy as np
import pytest

from _gpu_util import dev_fields
from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(32, 24, 16), (48, 16, 36)])
@pytest.mark.parametrize("top", [ppe.BC_WALL, ppe.BC_OUTFLOW])
def test_captured_projections(shape, top):
    import torch
    fl = fields.make_fields(*shape, seed=77, recipe="multimode", width=4.0, rho_g=60.0)
    d = dev_fields(fl)
    keep = {k: t.clone() for k, t in d.items()}
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    plans = [ppe.Plan(*shape, fl.lx, fl.ly, fl.lz, precision=p, bc_top=top, stream=main)
             for p in (ppe.FP64, ppe.FP32_REFINE)]

    def outs():
        return [torch.zeros_like(d[k]) for k in ("rho", "u", "v", "w")]

    def project(pl, o):
        pl.project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], fl.dt, *o)

    torch.cuda.synchronize()
    want = []
    for pl in plans:
        o = outs()
        with torch.cuda.stream(main):
            project(pl, o)
        torch.cuda.synchronize()
        want.append([t.cpu().numpy() for t in o])
    got = [outs() for _ in plans]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=main):
        side.wait_stream(main)
        with torch.cuda.stream(side):
            d["rho"].copy_(keep["rho"])
        d["u"].mul_(1.0)
        main.wait_stream(side)
        for pl, o in zip(plans, got):
            project(pl, o)
    for _ in range(2):
        for o in got:
            for t in o:
                t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for o, w in zip(got, want):
            for t, r in zip(o, w):
                assert np.array_equal(t.cpu().numpy(), r)
    for pl in plans:
        assert pl.info(allow_incompatible=True).f_max > 0
        pl.close()
