"""The right-hand side's column stacks at the edges of their tiling: widths
with and without an instance of their own, one or many stacks per CTA, tiles
that end past the top wall, one-plane chunks, and a rho_0 far above the density
(1 - rho_0/rho_f below -1).  The projection in FP64 against the numpy oracle,
bound 1e-12 relative: a few hundred pair operations of 2^-46 = 1.4e-14 each on
f, and the bound the solve is held to elsewhere."""
import numpy as np
import pytest

from _gpu_util import project_gpu
from oracle import ppe_oracle as O
from paper_2103_01874_gb300 import fields, ppe

pytestmark = pytest.mark.gpu

SHAPES = [(8, 27, 9), (16, 81, 8), (18, 8, 12), (32, 12, 9), (64, 27, 8), (96, 9, 16), (128, 18, 8), (144, 9, 8),
          (192, 9, 12), (256, 27, 8), (288, 8, 9), (384, 9, 8), (432, 9, 8), (512, 8, 9), (576, 9, 8)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("rule", [ppe.FACE_ARITHMETIC, ppe.FACE_HARMONIC])
@pytest.mark.parametrize("rho0", [-1.0, 2500.0])
def test_projection_at_tile_edges(shape, rule, rho0):
    nx, ny, nz = shape
    # spacings within a factor of two, so that the solve's own conditioning stays the usual one
    h = 2.0 * np.pi / ny
    fl = fields.make_fields(nx, ny, nz, seed=nx + ny, recipe="single", width=3.0, lx=0.8 * h * nx, lz=1.3 * h * nz)
    ref = O.project_fields(fl, rule=rule, rho0=rho0 if rho0 > 0 else None)
    res, _ = project_gpu(fl, face_rule=rule, rho0=rho0)
    for k in ("f", "p", "u", "v", "w"):
        assert np.isfinite(res[k]).all()
        assert O.rel_linf(res[k], ref[k]) <= 1e-12, k
