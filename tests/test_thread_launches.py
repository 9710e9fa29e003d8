"""Objects used from several host threads at once, each on its own stream.  Kernels
whose shared-memory tile varies from call to call are shared by all objects of a
process, so one thread's launch must not depend on the size the other asks for:
every call succeeds, and the results are those of a single thread (equal bits)."""
import threading

import pytest

from paper_2010_00409_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(torch, jobs):
    """Each job on a host thread of its own, all started together."""
    start, errors = threading.Barrier(len(jobs)), []

    def body(job):
        try:
            start.wait()
            job()
        except Exception as e:                      # noqa: BLE001 (reported below)
            errors.append(e)

    threads = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[0]


def _context(lib, torch, shape, prec, path):
    g = W.GridSpec(*shape, 0.5, 0.7, 0.3, 0.0, 0.0, 0.0, 1.0)
    ctx = lib.Context(g, None, 0.3, prec, stream=torch.cuda.Stream())
    ctx.set_kernel_path(path)
    ctx.set_fields(W.random_complex_field((6, shape[2], shape[1], shape[0]), seed=shape[0]))
    return ctx


# y tiles of 2 and 30 KB, k-space tiles of 5 and 92 KB, of the same kernels (radices up to 16)
@pytest.mark.parametrize("prec", [32, 64])
def test_run_time_passes_of_two_threads(lib, prec):
    import torch
    shapes, out = [(20, 16, 12), (16, 240, 240)], []
    n = 400
    for threads in (False, True):
        ctxs = [_context(lib, torch, s, prec, lib.PATH_GENERIC) for s in shapes]
        torch.cuda.synchronize()
        jobs = [lambda c=c: [c.advance(1) for _ in range(n)] for c in ctxs]
        if threads:
            _run(torch, jobs)
        else:
            for j in jobs:
                j()
        torch.cuda.synchronize()
        out.append([c.get_field(-1) for c in ctxs])
        for c in ctxs:
            c.close()
    for a, b in zip(*out):
        assert a.tobytes() == b.tobytes()


def test_batched_advances_of_two_threads(lib):
    import torch
    batches = [[_context(lib, torch, s, 32, lib.PATH_AUTO)] for s in ((18, 6, 6), (24, 96, 192))]
    torch.cuda.synchronize()
    _run(torch, [lambda b=b: [lib.multi_advance(b, 1) for _ in range(300)] for b in batches])
    for b in batches:
        b[0].synchronize()
        b[0].close()


# 77 and 102 KB of weight rows and spectra in the backward mixing kernel
def test_gradients_of_models_of_two_widths_in_four_threads(lib):
    import torch
    B, P, out = 4, 4, []
    prm = torch.linspace(-1, 1, 6 * B, device="cuda").view(B, 6).contiguous()
    tgt = torch.linspace(-1, 1, B * P ** 3, device="cuda").view(B, 1, P, P, P).contiguous()
    for threads in (False, True):
        nets = [lib.Fno(6, width=w, layers=4, patch=P, modes=1, hidden=8, out_channels=1, max_batch=B, seed=w,
                        stream=torch.cuda.Stream()) for w in (96, 128, 96, 128)]
        torch.cuda.synchronize()
        jobs = [lambda n=n: [n.loss_backward(prm, tgt, want_loss=False) for _ in range(400)] for n in nets]
        if threads:
            _run(torch, jobs)
        else:
            for j in jobs:
                j()
        torch.cuda.synchronize()
        out.append([n.grads.clone() for n in nets])
        for n in nets:
            n.close()
    for a, b in zip(*out):
        assert torch.equal(a, b)
