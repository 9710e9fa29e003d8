"""Focal-plane sampling of float32 storage at sizes off the kernels' tiles: rows
shorter than the eight lanes that share one, points and components that leave
partial 16 x 16 output tiles, sums that are no multiple of the 32-term chunk.
Tolerance as in the parity tests (float32 1e-5 on the oracle's plane)."""
import numpy as np
import pytest

from oracle import psatd_oracle as O
from paper_2010_00409_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,ny,nz,comps", [((1, 1, 1), 1, 1, (0,)), ((3, 5, 2), 2, 17, (5,)),
                                               ((9, 36, 25), 16, 15, (0, 4)), ((25, 32, 64), 33, 1, (0, 1, 2)),
                                               ((64, 8, 45), 48, 40, (0, 1, 2, 3, 4, 5))])
def test_float32_planes_match_oracle(lib, shape, ny, nz, comps):
    nx, nyg, nzg = shape
    g = W.GridSpec(nx, nyg, nzg, 0.5, 0.7, 0.3, -0.25 * nx, -0.35 * nyg, -0.15 * nzg, 1.0)
    f = W.random_complex_field((6, nzg, nyg, nx), seed=nx)
    m = W.MappingSpec(R0=4.0, L=1e3)                      # a shell that cuts nothing
    args = (0.013, ny, nz, -0.31 * nyg, 0.29 * nyg, -0.11 * nzg, 0.13 * nzg)
    with lib.Context(g, m, 0.1, 32) as ctx:
        ctx.set_fields(f)
        ctx.set_time(4.0)
        got = ctx.sample_focal_plane(*args, comps=comps)
    f32 = f.astype(np.complex64).astype(np.complex128)
    og = O.Grid(nx, nyg, nzg, g.dx, g.dy, g.dz, g.x_min, g.y_min, g.z_min, g.c)
    ys = args[3] + (args[4] - args[3]) * np.arange(ny) / ny
    zs = args[5] + (args[6] - args[5]) * np.arange(nz) / nz
    ref = O.sample_plane(f32, og, O.Mapping(m.R0, m.L), args[0], ys, zs, 4.0, comps=comps)
    ref = np.asarray(ref)
    assert got.shape == ref.shape
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
