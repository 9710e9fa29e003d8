"""The staging GEMM on both sides of the line between one block of 512 threads per SM
(no more tiles than SMs) and several of 256: tiles of 32, 64 and 128 columns, K blocks
with a remainder, split K, C added to.  Against float64 products of the operands rounded
to bfloat16: float32 accumulation of K products stays within K 2^-24 of the sum of the
magnitudes (and of C's)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K,ksplit,beta", [
    (1, 1, 1, 1, 0.0), (128, 32, 64, 1, 0.5), (130, 33, 65, 1, 0.0), (127, 128, 520, 1, 1.0), (300, 20, 1000, 4, 0.25),
    (128 * 152, 17, 40, 1, 0.5), (128 * 152 + 1, 17, 40, 1, 0.5), (128 * 76, 120, 200, 2, 0.0), (128 * 77, 120, 200, 2, 0.0),
    (128 * 151 + 5, 64, 72, 1, 0.0)])
@pytest.mark.parametrize("ta,tb,tc", [(0, 0, 0), (0, 1, 1), (1, 0, 1)])
def test_products_on_both_sides_of_the_line(lib, M, N, K, ksplit, beta, ta, tb, tc):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M + N + K)

    def mat(a, b, t):
        x = torch.randn((b, a) if t else (a, b), generator=g, device="cuda")
        return x.t() if t else x

    A, B, C = mat(M, K, ta), mat(K, N, tb), mat(M, N, tc)
    a, b, c = (x.to(torch.float64) for x in (A.to(torch.bfloat16), B.to(torch.bfloat16), C))
    want, size = 0.5 * (a @ b) + beta * c, 0.5 * (a.abs() @ b.abs()) + abs(beta) * c.abs()
    lib.gemm_bf16(A, B, C, alpha=0.5, beta=beta, ksplit=ksplit)
    lib.gemm_synchronize()
    assert bool(((C.to(torch.float64) - want).abs() <= (K + ksplit + 4) * 2.0 ** -24 * size + 1e-30).all())
