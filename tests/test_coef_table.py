"""The per-mode coefficient table built on the device: steps of new sizes after
psatd_set_dt against the oracle at lengths with and without a Nyquist mode, and
the refusal under stream capture.  Tolerance: one step of the parity tests
(float64 1e-12, float32 1e-5)."""
import numpy as np
import pytest

from oracle import psatd_oracle as O
from paper_2010_00409_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 4, 9), (2, 15, 1), (32, 6, 25)])
@pytest.mark.parametrize("prec,tol", [(64, 1e-12), (32, 1e-5)])
def test_new_steps_match_oracle(lib, shape, prec, tol):
    nx, ny, nz = shape
    g = W.GridSpec(nx, ny, nz, 0.5, 0.7, 0.3, 0.0, 0.0, 0.0, 1.3)
    og = O.Grid(nx, ny, nz, g.dx, g.dy, g.dz, 0.0, 0.0, 0.0, g.c)
    f = W.random_complex_field((6, nz, ny, nx), seed=nx + 10 * ny)
    with lib.Context(g, None, 0.1, prec) as ctx:
        for dt in (0.37, -1.9, 0.0, 250.0):
            ctx.set_fields(f)
            ctx.set_dt(dt)
            ctx.advance(1)
            got = ctx.get_field(-1)
            ref = O.advance(f, og, dt, 1)
            assert np.linalg.norm(got - ref) <= tol * np.linalg.norm(ref), dt


def test_new_table_is_refused_under_capture(lib):
    import torch
    g = W.GridSpec(8, 8, 8, 0.5, 0.7, 0.3, 0.0, 0.0, 0.0, 1.0)
    s = torch.cuda.Stream()
    with lib.Context(g, None, 0.1, 32, stream=s) as ctx:
        b = lib.Batch(s)
        with b:
            ctx.advance(1)
            with pytest.raises(lib.PsatdError):
                ctx.set_dt(0.2)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s, capture_error_mode="thread_local"):
            with pytest.raises(lib.PsatdError):
                ctx.set_dt(0.2)                        # a capture the library did not begin
        b.close()
