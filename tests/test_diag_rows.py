"""Diagnostics of random (not divergence-free) fields at row lengths around the
blocks' split into rows: one value, rows that leave spare threads, one row of a block
and a row longer than a block, against the oracle.  The maxima come from transforms
good to 1e-5 (float32) and 1e-12 (float64) of the field's norm; a maximum over n modes
is at least norm / sqrt(n) up to a factor of order one, so it is held to that times
sqrt(n)."""
import numpy as np
import pytest

from oracle import psatd_oracle as O
from paper_2010_00409_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 8, 6), (5, 6, 9), (64, 4, 5), (100, 3, 8), (250, 6, 2), (256, 3, 4), (270, 4, 3)])
@pytest.mark.parametrize("prec,tol", [(64, 1e-12), (32, 1e-5)])
def test_maxima_match_oracle_at_every_row_split(lib, shape, prec, tol):
    nx, ny, nz = shape
    g = W.GridSpec(nx, ny, nz, 0.5, 0.7, 0.3, 0.0, 0.0, 0.0, 1.0)
    f = W.random_complex_field((6, nz, ny, nx), seed=nx)
    want = O.diagnostics(f, O.Grid(nx, ny, nz, g.dx, g.dy, g.dz, 0.0, 0.0, 0.0, 1.0))
    with lib.Context(g, None, 0.3, prec) as ctx:
        ctx.set_fields(f)
        got = ctx.diagnostics()
    for k in ("energy_E", "energy_B", "max_div_E", "max_div_B", "max_E_hat", "max_B_hat"):
        assert abs(got[k] - want[k]) <= tol * np.sqrt(nx * ny * nz) * want[k], k
