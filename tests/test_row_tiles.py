"""x axes whose row tiles differ: the padded shared-memory layout (float32 plans of three
levels with a last radix of 8: 2048 = 16 x 16 x 8, 1536, 1280, 1152), float64 tiles
widened to fill their warps (1000, 480, 60, 25) and neighbours of both, with a remainder
of rows in the last tile: forward and inverse transform against numpy (parity
tolerances)."""
import numpy as np
import pytest

from paper_2010_00409_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [2048, 1920, 1536, 1280, 1152, 1024, 1000, 480, 108, 60, 25, 4])
@pytest.mark.parametrize("ny,nz", [(1, 1), (5, 3)])
@pytest.mark.parametrize("prec,tol", [(32, 1e-5), (64, 1e-12)])
@pytest.mark.parametrize("path", ["PATH_AUTO", "PATH_GENERIC"])
def test_rows_match_numpy(lib, nx, ny, nz, prec, tol, path):
    g = W.GridSpec(nx, ny, nz, 0.5, 0.7, 0.3, 0.0, 0.0, 0.0, 1.0)
    f = W.random_complex_field((6, nz, ny, nx), seed=nx)
    F = np.fft.fftn(f, axes=(1, 2, 3))
    with lib.Context(g, None, 0.3, prec) as ctx:
        ctx.set_kernel_path(getattr(lib, path))
        ctx.set_fields(f)
        ctx.fft(lib.FORWARD)
        assert np.linalg.norm(ctx.get_field(-1) - F) <= tol * np.linalg.norm(F)
        ctx.fft(lib.INVERSE)
        assert np.linalg.norm(ctx.get_field(-1) / g.cells - f) <= 2 * tol * np.linalg.norm(f)
