"""The surrogate's bias gradients are sums over every voxel; the reduction has to lose
nothing that a float64 sum of the same float32 values keeps.

With all weights zero but the last layer's (and its values powers of two) the
pre-activations are zero, so gelu'(0) = 1/2 and the summed values are known in full:
the loss gradient g = 2 (out - target) / n of the output bias and bfloat16(g) w / 2 of
the projection bias (its contraction rounds g to bfloat16)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _gradients(lib, torch, P, B, w, tgt):
    """(output bias, projection bias) gradients of a model with last-layer weights w."""
    H = len(w)
    net = lib.Fno(1, width=1, layers=1, patch=P, modes=1, hidden=H, out_channels=1, max_batch=B, seed=0)
    net.params.zero_()
    net.params[-1 - H:-1] = torch.tensor(w, dtype=torch.float32, device="cuda")
    net.loss_backward(torch.zeros((B, 1), device="cuda"), torch.tensor(tgt, device="cuda"), want_loss=False)
    g = net.grads.cpu().numpy()
    net.close()
    return g[-1], g[-1 - 2 * H:-1 - H]


def _pieces(total, k):
    """k integers of at most eight significant bits each that sum to total."""
    out = []
    for _ in range(k):
        s = max(abs(total).bit_length() - 8, 0)
        p = (abs(total) >> s << s) * (1 if total >= 0 else -1)
        out.append(p)
        total -= p
    assert total == 0
    return out


@pytest.mark.parametrize("seed", range(4))
def test_sums_keep_53_bits(lib, seed):
    """32 values that one thread adds: integers of eight bits times powers of two whose
    partial sums stay below 2^53, so that float64 adds them exactly in any order, and
    whose large parts cancel.  A sum of 48 bits is off by units."""
    import torch
    P, rest = 64, 12345
    rng = np.random.default_rng(seed)
    v = [int(rng.integers(128, 256) | 1) << int(e) for e in np.linspace(44.9, 0, 22)]
    v += _pieces(rest - sum(v), 10)
    assert len(v) == 32 and all(abs(sum(v[:i])) < 2 ** 53 for i in range(33))
    n = P ** 3
    t = np.zeros(n, np.float32)
    for k in range(8):
        t[1024 * k:1024 * k + 4] = v[4 * k:4 * k + 4]          # voxels of the first chunk's first thread
    out, proj = _gradients(lib, torch, P, 1, [1.0], t.reshape(1, 1, P, P, P))
    assert out == -2.0 * rest / n
    assert proj[0] == -1.0 * rest / n


@pytest.mark.parametrize("values,want", [((np.inf,), -np.inf), ((-np.inf, 1.0), np.inf), ((np.inf, -np.inf), np.nan),
                                         ((np.nan, np.inf), np.nan)])
def test_infinities_stay_infinities(lib, values, want):
    import torch
    P = 8
    t = np.ones(P ** 3, np.float32)
    t[37:37 + 5 * len(values):5] = values
    out, proj = _gradients(lib, torch, P, 1, [1.0], t.reshape(1, 1, P, P, P))
    np.testing.assert_equal(np.array([out, proj[0]], np.float64), [want, want])


@pytest.mark.parametrize("P,B,w", [(4, 1, [1.0]), (6, 3, [1.0, -0.5, 2.0]), (10, 2, [0.25, 4.0]), (36, 5, [1.0, 2.0])])
def test_every_bias_equals_its_float64_sum(lib, P, B, w):
    """Patches whose voxels leave chunks empty or uneven.  The sum's error against
    float64 and its rounding to float32 stay below 2^-22 of the sum of magnitudes."""
    import torch
    rng = np.random.default_rng(P)
    t = (rng.standard_normal((B, 1, P, P, P)) + 0.5).astype(np.float32)
    out, proj = _gradients(lib, torch, P, B, w, t)
    g = np.float32(2) * (np.float32(0) - t) / np.float32(t.size)
    assert abs(out - g.sum(dtype=np.float64)) <= 2.0 ** -22 * np.abs(g).sum(dtype=np.float64)
    gb = torch.tensor(g).to(torch.bfloat16).to(torch.float64).numpy()
    for have, x in zip(proj, w):
        want = 0.5 * x * gb
        assert abs(have - want.sum()) <= 2.0 ** -22 * np.abs(want).sum()
