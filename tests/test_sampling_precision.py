"""The double-float sums of focal-plane sampling (float32 storage) over the longest
axis: no further from their exact value than one chain of renormalised double-float
sums over the row (each product and each sum rounded to a normalised pair), which is
evaluated here in float32.

Samples are float32, so the sums are made to cancel: products of one sign over the
row, and two values that bring the exact sum to about 2^-48 of the sum of magnitudes.
The other two axes are sampled on their nodes, where their weights are 0 and 1."""
import numpy as np
import pytest

from paper_2010_00409_gb300 import workloads as W

pytestmark = pytest.mark.gpu

f4 = np.float32
N, K = 2048, 64


def _two_sum(a, b):
    s = a + b
    t = s - a
    return s, (a - (s - t)) + (b - t)


def _quick(a, b):
    s = a + b
    return s, b - (s - a)


def _add(a, b):
    s, e = _two_sum(a[0], b[0])
    return _quick(s, e + (a[1] + b[1]))


def _mul(w, v):
    p = w[0] * v
    d = np.float64
    e = (d(w[0]) * v - p).astype(f4)
    return _quick(p, (d(w[1]) * v + e).astype(f4))


def _weights(points):
    """w_N(s) of the trigonometric interpolant at unit spacing, complex128 [points][N]."""
    u = (points[:, None] - np.arange(N)) / N
    u = u - np.floor(u + 0.5)

    def sinpi(x):
        r = x - 2 * np.round(x / 2)                          # exact for the dyadic points used here
        return np.sin(np.pi * np.where(np.abs(r) > 0.5, np.sign(r) - r, r))

    ratio = sinpi(N * u) / (N * sinpi(u))
    a = 2 * (-(N // 2) + 0.5 * (N - 1)) * u
    return ratio * (sinpi(a + 0.5) + 1j * sinpi(a))


def _rows(w, rng):
    """Rows v [6][K][N] (complex64) for the weights w [K][N]: the real part of their sum cancels."""
    r = rng.uniform(0.2, 1.0, (2, 6, K, N)) / np.abs(w)
    v = (r[0] * np.sign(w.real) - 1j * r[1] * np.sign(w.imag)).astype(np.complex64)
    big = np.argsort(-np.abs(w.real), axis=-1)
    rows = np.arange(K)
    for j in (big[:, 0], big[:, 1]):
        s = _exact(w, v) - w.real[rows, j] * v.real[:, rows, j].astype(np.longdouble)
        v.real[:, rows, j] = (-s / w.real[rows, j]).astype(f4)
    return v


def _terms(w, v):
    l = np.longdouble
    return w.real.astype(l) * v.real, -(w.imag.astype(l) * v.imag)


def _exact(w, v):
    return sum(t.sum(axis=-1) for t in _terms(w, v))


def _chain(w, v):
    """One chain of renormalised double-float sums (real part), rounded to float32."""
    def pair(x):
        h = x.astype(f4)
        return h, (x - h).astype(f4)

    wr, wi = pair(w.real), pair(w.imag)
    z = np.zeros(v.shape[:-1], f4)
    acc = (z, z)
    for j in range(N):
        at = (Ellipsis, j)
        m = _mul((-wi[0][at], -wi[1][at]), v.imag[at])
        acc = _add(acc, _add(_mul((wr[0][at], wr[1][at]), v.real[at]), m))
    return acc[0] + acc[1]


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_sums_over_an_axis_keep_their_bits(lib, axis):
    rng = np.random.default_rng(axis)
    shape = {0: (N, K, 1), 1: (1, N, K), 2: (1, K, N)}[axis]
    step, first = (0.0, 731.40625) if axis == 0 else (31.0, 0.40625)
    points = first + step * np.arange(K)
    w = _weights(points)
    v = _rows(w, rng)
    f = {0: v[:, None], 1: v[..., None], 2: v.transpose(0, 2, 1)[..., None]}[axis]
    g = W.GridSpec(*shape, 1.0, 1.0, 1.0, 0.0, 0.0, 0.0, 1.0)
    m = W.MappingSpec(R0=1e5, L=1e6)                         # a shell that cuts nothing
    node, pts = (0.0, float(K)), (first, first + step * K)
    with lib.Context(g, m, 0.1, 32) as ctx:
        ctx.set_fields(np.ascontiguousarray(f.astype(np.complex64)))
        ctx.set_time(1e5)
        if axis == 0:
            got = ctx.sample_focal_plane(first, K, 1, *node, 0.0, 1.0, comps=range(6))[:, 0]
        else:
            lim = (pts + node) if axis == 1 else (node + pts)
            got = ctx.sample_focal_plane(0.0, K, K, *lim, comps=range(6))
            got = np.diagonal(got, axis1=1, axis2=2)
    exact, mag = _exact(w, v), sum(np.abs(t).sum(axis=-1) for t in _terms(w, v))
    assert np.all(np.abs(exact) < 1e-10 * mag)
    err = np.asarray((got.real - exact) / mag, float)
    old = np.asarray((_chain(w, v) - exact) / mag, float)
    assert np.sqrt(np.mean(err ** 2)) <= np.sqrt(np.mean(old ** 2)), (np.abs(err).max(), np.abs(old).max())
