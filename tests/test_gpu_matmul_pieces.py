"""Binary32 products on the tensor cores: what the three bf16 pieces of an
operand and the two accumulators must give where few terms meet, through the C ABI
against binary64.  Sizes take each tile form (128 x 64, 128 x 128, a CTA pair's
256 x 256), with remainders, an odd count of 32-deep chunks, and sums over the end of
an accumulation of the smaller products (2048 k, a pair's 8192 k)."""
import numpy as np
import pytest

from test_gpu_matmul_split import env, product   # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1000, 1000, 1000), (1537, 1023, 2049), (2000, 2040, 1111),
                                   (2048, 2048, 2048), (2000, 2040, 9000)])
def test_one_term_per_entry(env, shape):   # noqa: F811
    """One non-zero entry in each row of A: every entry is a single product,
    with all the pieces' products in it.  At most 2^-24 of it is left out
    (|x2| <= 2^-8 |x|, |x3| <= 2^-17 |x|: x2 y3 + x3 y2 <= 2^-24, x3 y3 2^-34), the
    smaller products' sum (2^-7) is truncated five times at 2^-23, and the whole is
    rounded once at 2^-24: 2.25 x 2^-24.  On average the rounding is all there is:
    uniform in +-2^-24 at most, 2^-24 / sqrt 3 by its square, and without a sign
    (mean of 10^6 entries: 10^-3 of the deviation)."""
    _, _, torch = env
    M, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(K)
    A = torch.zeros(M, K, device="cuda")
    A[torch.arange(M, device="cuda"), torch.randint(0, K, (M,), device="cuda", generator=g)] = \
        torch.randn(M, device="cuda", generator=g)
    B = torch.randn(K, N, device="cuda", generator=g)
    ref = A.double() @ B.double()
    C = torch.from_numpy(product(env, A, B)).cuda().double()
    zero = ref == 0.0
    assert not C[zero].any()
    rel = ((C - ref) / ref)[~zero] * 2.0 ** 24
    assert float(rel.abs().max()) <= 2.25
    assert float(rel.square().mean().sqrt()) <= 0.6
    assert abs(float(rel.mean())) <= 0.02


@pytest.mark.parametrize("side", [0, 1])
@pytest.mark.parametrize("shape", [(1000, 1000, 300), (1000, 1000, 1000), (700, 900, 2049),
                                   (700, 900, 4100), (1537, 1023, 2049), (2000, 2040, 160),
                                   (2000, 2040, 1111)])
def test_three_pieces_times_signs(env, shape, side):   # noqa: F811
    """x = p + q 2^-9 + r 2^-17 with 64 <= |p|, |q| < 128 and |r| < 64: the pieces
    are p, q 2^-9 and r 2^-17.  Times +-1, dense: the sums of p and of the others are
    exact (below 2^24 of their last bits), so the product is the exact one rounded
    once."""
    _, _, torch = env
    M, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(M + N + K + side)

    def signed(lo, hi, *s):
        v = torch.randint(lo, hi, s, device="cuda", generator=g).float()
        return v * (torch.randint(0, 2, s, device="cuda", generator=g) * 2 - 1)
    s = (M, K) if side == 0 else (K, N)
    x = signed(64, 128, *s) + signed(64, 128, *s) * 2.0 ** -9
    x += signed(0, 64, *s) * 2.0 ** -17
    e = signed(1, 2, *((K, N) if side == 0 else (M, K)))
    A, B = (x, e) if side == 0 else (e, x)
    ref = (A.double() @ B.double()).cpu().numpy().astype(np.float32)
    assert np.array_equal(product(env, A, B), ref)
