"""The mixed-radix axis transforms (run-time passes and the compile-time two-pass
kernels) at lengths whose plans differ in passes and radices, with x extents off
the 16- and 8-column tiles: forward and inverse transforms and one step against
the oracle.  The GENERIC path runs the run-time passes, AUTO the compile-time
ones where a length has them; both have to agree with the oracle within the
parity tolerances (float64 1e-12, float32 1e-5)."""
import numpy as np
import pytest

from oracle import psatd_oracle as O
from paper_2010_00409_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# two-pass plans (18 = 6 x 3 ... 240 = 16 x 15), wide radices (162 = 18 x 9, 243 = 27 x 9,
# 480 = 24 x 20), three passes in float64 (162, 243) and in both (1000), one pass, N = 1
SHAPES = [(18, 27, 20), (25, 36, 162), (45, 1, 96), (50, 243, 3), (75, 16, 60), (135, 12, 10), (9, 240, 5),
          (100, 2, 81), (480, 3, 2), (2, 480, 3), (3, 2, 480), (4, 1000, 2), (1000, 2, 3), (8, 4, 1000),
          (162, 5, 225)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prec,tol", [(64, 1e-12), (32, 1e-5)])
@pytest.mark.parametrize("path", ["PATH_AUTO", "PATH_GENERIC"])
def test_transforms_and_step_match_oracle(lib, shape, prec, tol, path):
    nx, ny, nz = shape
    g = W.GridSpec(nx, ny, nz, 0.5, 0.7, 0.3, 0.0, 0.0, 0.0, 1.0)
    og = O.Grid(nx, ny, nz, g.dx, g.dy, g.dz, 0.0, 0.0, 0.0, 1.0)
    f = W.random_complex_field((6, nz, ny, nx), seed=nx + ny)
    F = np.fft.fftn(f, axes=(1, 2, 3))
    with lib.Context(g, None, 0.3, prec) as ctx:
        ctx.set_kernel_path(getattr(lib, path))
        ctx.set_fields(f)
        ctx.fft(lib.FORWARD)
        got = ctx.get_field(-1)
        assert np.linalg.norm(got - F) <= tol * np.linalg.norm(F)
        ctx.fft(lib.INVERSE)
        got = ctx.get_field(-1) / g.cells
        assert np.linalg.norm(got - f) <= 2 * tol * np.linalg.norm(f)
        ctx.set_fields(f)
        ctx.advance(1)
        got = ctx.get_field(-1)
    ref = O.advance(f, og, 0.3, 1)
    assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref)


def test_every_compile_time_length_matches_the_run_time_passes(lib):
    """The compile-time kernels of every length against the run-time passes of the
    same plan, along x, y and z (float32, same arithmetic order: 1e-6)."""
    lengths = [n for n in range(18, 1025) if any(n == 2 ** a * 3 ** b * 5 ** c for a in range(9) for b in range(6)
                                                for c in range(4))]
    for n in lengths:
        for shape in ((n, 2, 1), (18, n, 1), (18, 1, n)) if n > 256 else ((n, 3, 4), (18, n, 2), (18, 3, n)):
            nx, ny, nz = shape
            g = W.GridSpec(nx, ny, nz, 0.5, 0.7, 0.3, 0.0, 0.0, 0.0, 1.0)
            f = W.random_complex_field((6, nz, ny, nx), seed=n)
            out = []
            for path in (lib.PATH_AUTO, lib.PATH_GENERIC):
                with lib.Context(g, None, 0.3, 32) as ctx:
                    ctx.set_kernel_path(path)
                    ctx.set_fields(f)
                    ctx.advance(1)
                    out.append(ctx.get_field(-1))
            assert np.linalg.norm(out[0] - out[1]) <= 1e-6 * np.linalg.norm(out[1]), shape


@pytest.mark.parametrize("shape", [(6, 512, 2), (18, 2, 512), (36, 1024, 1), (16, 1, 1024), (512, 3, 64), (512, 2, 512)])
def test_three_pass_columns_and_row_fused_steps_match_oracle(lib, shape):
    """512- and 1024-point y and z transforms over column tiles of 16 with a
    remainder, and the row-fused step at N_x = 512 on a z length that also has a
    fused z pass (float32, parity tolerance 1e-5)."""
    nx, ny, nz = shape
    g = W.GridSpec(nx, ny, nz, 0.5, 0.7, 0.3, 0.0, 0.0, 0.0, 1.0)
    f = W.random_complex_field((6, nz, ny, nx), seed=ny)
    with lib.Context(g, None, 0.3, 32) as ctx:
        ctx.set_fields(f)
        ctx.advance(1)
        got = ctx.get_field(-1)
    ref = O.advance(f, O.Grid(nx, ny, nz, g.dx, g.dy, g.dz, 0.0, 0.0, 0.0, 1.0), 0.3, 1)
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)


def test_batched_compile_time_tiles_match_the_run_time_passes(lib):
    """One batched launch over boxes with every length of two radices up to 16 along
    x, y and z (remainders of all three tiles) against the run-time passes of a
    context each (float32, same arithmetic order: 1e-6)."""
    lengths = [n for n in range(18, 257) if any(n == 2 ** a * 3 ** b * 5 ** c for a in range(9) for b in range(6)
                                               for c in range(4))]
    ctxs, want = [], []
    for n in lengths:
        for shape in ((n, 3, 5), (18, n, 2), (20 if n % 2 else 10, 3, n)):
            nx, ny, nz = shape
            g = W.GridSpec(nx, ny, nz, 0.5, 0.7, 0.3, 0.0, 0.0, 0.0, 1.0)
            f = W.random_complex_field((6, nz, ny, nx), seed=n)
            with lib.Context(g, None, 0.3, 32) as ctx:
                ctx.set_kernel_path(lib.PATH_GENERIC)
                ctx.set_fields(f)
                ctx.advance(1)
                want.append(ctx.get_field(-1))
            ctxs.append(lib.Context(g, None, 0.3, 32))
            ctxs[-1].set_fields(f)
    lib.multi_advance(ctxs, 1)
    for ctx, w in zip(ctxs, want):
        got = ctx.get_field(-1)
        assert np.linalg.norm(got - w) <= 1e-6 * np.linalg.norm(w), w.shape
        ctx.close()
