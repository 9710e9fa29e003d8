"""The x contraction of focal-plane sampling on both sides of its line between 8 and 32
lanes a row: few long rows, rows that are no multiple of either, real fields of one
component and of six.  Tolerance as in the parity tests (float32 1e-5 on the oracle's
plane)."""
import numpy as np
import pytest

from oracle import psatd_oracle as O
from paper_2010_00409_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _check(lib, g, ctx, f, comps, ny, nz):
    m = W.MappingSpec(R0=4.0, L=1e3)                      # a shell that cuts nothing
    ctx.set_fields(f)
    ctx.set_time(4.0)
    args = (0.013, ny, nz, -0.31 * g.Ny, 0.29 * g.Ny, -0.11 * g.Nz, 0.13 * g.Nz)
    got = ctx.sample_focal_plane(*args, comps=comps)
    og = O.Grid(g.Nx, g.Ny, g.Nz, g.dx, g.dy, g.dz, g.x_min, g.y_min, g.z_min, g.c)
    ys = args[3] + (args[4] - args[3]) * np.arange(ny) / ny
    zs = args[5] + (args[6] - args[5]) * np.arange(nz) / nz
    ref = np.asarray(O.sample_plane(f.astype(np.complex128), og, O.Mapping(m.R0, m.L), args[0], ys, zs, 4.0, comps=comps))
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


def _grid(nx, ny, nz):
    return W.GridSpec(nx, ny, nz, 0.5, 0.7, 0.3, -0.25 * nx, -0.35 * ny, -0.15 * nz, 1.0)


@pytest.mark.parametrize("shape,comps", [((125, 5, 3), (0,)), ((128, 4, 1), (0, 5)), ((135, 3, 8), (0, 1, 2)),
                                         ((1000, 2, 3), (0, 1, 2, 3, 4, 5)), ((135, 81, 40), (0, 1, 2, 3, 4, 5))])
def test_complex_rows_match_oracle(lib, shape, comps):
    g = _grid(*shape)
    f = W.random_complex_field((6, g.Nz, g.Ny, g.Nx), seed=g.Nx).astype(np.complex64)
    with lib.Context(g, W.MappingSpec(R0=4.0, L=1e3), 0.1, 32) as ctx:
        _check(lib, g, ctx, f, comps, 5, 4)


@pytest.mark.parametrize("comps", [(0,), (0, 1, 2, 3, 4, 5)])
def test_real_rows_match_oracle(lib, comps):
    g = _grid(256, 256, 64)
    f = np.random.default_rng(3).standard_normal((6, g.Nz, g.Ny, g.Nx)).astype(np.float32)
    with lib.Context(g, W.MappingSpec(R0=4.0, L=1e3), 0.1, 32, real=True) as ctx:
        _check(lib, g, ctx, f, comps, 3, 4)
