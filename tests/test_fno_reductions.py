"""The surrogate's gradient reductions at sizes off their tiles: channels that
leave partial 32 x 32 weight tiles, patches whose voxel count is no multiple of the
16-voxel run (P = 6, 10: P^3 = 8 mod 16), batches that are no multiple of four.

The gradients of the pointwise layers are checked against float64 sums formed from
the model's own arrays: with a network of one spectral layer whose spectral weights
are zero, out = Wq2 gelu(Wq1 v1 + bq1) + bq2, v1 = W v0 + b, v0 = Wl f + bl.
Tolerance: the operands are rounded to bfloat16 (relative 2^-9 each); a bias
gradient is a sum of entries that passed two to three such contractions, so the
relative error of every gradient block stays below 3 %, the bound of the parity
tests of the network's gradients."""
import numpy as np
import pytest

from oracle import fno_oracle as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cfg,B", [((2, 5, 1, 6, 2, 7, 3), 1), ((6, 33, 1, 10, 3, 40, 3), 3),
                                   ((1, 32, 2, 8, 4, 64, 1), 5)])
def test_gradients_match_float64_autograd(lib, cfg, B):
    import torch
    c = F.FnoConfig(*cfg)
    net = lib.Fno(c.NP, width=c.C, layers=c.L, patch=c.P, modes=c.m, hidden=c.H, out_channels=c.NO, max_batch=B,
                  seed=3)
    rng = np.random.default_rng(5)
    theta = 0.3 * rng.standard_normal(F.num_params(c))
    prm = rng.uniform(-1, 1, (B, c.NP))
    tgt = rng.standard_normal((B, c.NO, c.P, c.P, c.P))
    net.params.copy_(torch.tensor(theta, dtype=torch.float32))
    net.loss_backward(torch.tensor(prm, dtype=torch.float32, device="cuda"),
                      torch.tensor(tgt, dtype=torch.float32, device="cuda"))
    got = net.grads.cpu().numpy().astype(np.float64)

    t = torch.tensor(theta, requires_grad=True)
    P, m, C = c.P, c.m, c.C
    o = [0]

    def take(*shape):
        n = int(np.prod(shape))
        v = t[o[0]:o[0] + n].reshape(shape)
        o[0] += n
        return v

    x = -1 + 2 * torch.arange(P, dtype=torch.float64) / P
    grid = torch.stack([x[None, None, :].expand(P, P, P), x[None, :, None].expand(P, P, P),
                        x[:, None, None].expand(P, P, P)])
    p = torch.tensor(prm)
    feat = torch.cat([p[:, :, None, None, None].expand(B, c.NP, P, P, P), grid[None].expand(B, 3, P, P, P)], 1)
    mix = lambda w, v: torch.einsum("oi,bizyx->bozyx", w, v)  # noqa: E731
    bias = lambda b: b[None, :, None, None, None]  # noqa: E731
    blocks = []
    s = o[0]
    v = mix(take(C, c.NP + 3), feat) + bias(take(C))
    blocks.append((s, o[0]))
    keep = torch.cat([torch.arange(m), torch.arange(P - m, P)])
    for l in range(c.L):
        s = o[0]
        R = take(2, 2 * m, 2 * m, m, C, C)
        sp = torch.fft.rfftn(v, dim=(-3, -2, -1))[..., :m].index_select(2, keep).index_select(3, keep)
        sp = torch.einsum("bizyx,zyxio->bozyx", sp, torch.complex(R[0], R[1]))
        full = torch.zeros((B, C, P, 2 * m, m), dtype=sp.dtype).index_copy(2, keep, sp)
        full = torch.zeros((B, C, P, P, m), dtype=sp.dtype).index_copy(3, keep, full)
        full = torch.cat([full, torch.zeros((B, C, P, P, P // 2 + 1 - m), dtype=sp.dtype)], -1)
        z = torch.fft.irfftn(full, s=(P, P, P), dim=(-3, -2, -1))
        blocks.append((s, o[0]))
        s = o[0]
        z = z + mix(take(C, C), v) + bias(take(C))
        blocks.append((s, o[0]))
        v = torch.nn.functional.gelu(z) if l + 1 < c.L else z
    s = o[0]
    h = torch.nn.functional.gelu(mix(take(c.H, C), v) + bias(take(c.H)))
    blocks.append((s, o[0]))
    s = o[0]
    out = mix(take(c.NO, c.H), h) + bias(take(c.NO))
    blocks.append((s, o[0]))
    ((out - torch.tensor(tgt)) ** 2).mean().backward()
    want = t.grad.numpy()
    assert np.all(np.isfinite(got))
    for a, b in blocks:
        assert np.linalg.norm(got[a:b] - want[a:b]) <= 0.03 * np.linalg.norm(want[a:b]), (a, b)
