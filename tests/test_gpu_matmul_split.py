"""Binary32 products on the tensor cores (operands in three bf16 pieces): the
tile forms' edges, the range of operands they take, and the CUDA-core form
that takes over outside it, through the C ABI against binary64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_6685_gb300 import safegpu as sg
    ctx = sg.sg_init(0, torch.cuda.current_stream().cuda_stream)
    yield sg, ctx, torch
    sg.sg_destroy(ctx)


def product(env, A, B):
    sg, ctx, _ = env
    ma, mb = sg.wrap_tensor(ctx, A), sg.wrap_tensor(ctx, B)
    mc = sg.sg_matmul(ctx, ma, mb, sg.SG_PREC_F32_SIMT)
    C = sg.sg_matrix_read(ctx, mc, np.empty((A.shape[0], B.shape[1]), np.float32))
    for h in (mc, ma, mb):
        sg.sg_matrix_release(h)
    return C


def bound(A, B):
    """Per entry: what the pieces leave out (2^-25.9), at most 32 truncations
    of a 32-deep sum at 2^-23, and one rounding at 2^-24 per 32 k added to the
    running sum (the CUDA cores' bound, K 2^-24, where that is larger)."""
    K = A.shape[1]
    u = max(2.0 ** -25.9 + 32 * 2.0 ** -23 + -(-K // 32) * 2.0 ** -24, K * 2.0 ** -24)
    return (A.double().abs() @ B.double().abs()).mul_(u).cpu().numpy()


# tiles of 128 x 64, 128 x 128 and 256 x 256 with remainders in each
# direction, K at and beside the 32- and 64-deep stages, odd leading dimensions
@pytest.mark.parametrize("shape", [(200, 200, 200), (129, 65, 1000), (1, 700, 3000),
                                   (700, 1, 3000), (513, 260, 97), (384, 384, 991),
                                   (1500, 1500, 160), (1531, 1409, 129), (2048, 2048, 96),
                                   (2049, 2303, 1023)])
@pytest.mark.parametrize("dist", ["normal", "uniform", "wide"])
def test_split_product(env, shape, dist):
    _, _, torch = env
    M, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(M + 3 * N + 7 * K)

    def draw(r, c):
        if dist == "uniform":
            return torch.rand(r, c, device="cuda", generator=g)
        x = torch.randn(r, c, device="cuda", generator=g)
        if dist == "wide":   # exponents over 2^-20 .. 2^20, some entries zero
            x = x * torch.exp2(torch.randint(-20, 21, (r, c), device="cuda", generator=g).float())
            x[torch.rand(r, c, device="cuda", generator=g) < 0.1] = 0.0
        return x
    A, B = draw(M, K), draw(K, N)
    C = product(env, A, B)
    ref = (A.double() @ B.double()).cpu().numpy()
    assert np.all(np.abs(C - ref) <= bound(A, B))


def test_split_integers_exact(env):
    """Integer products whose partial sums stay below 2^24 are exact."""
    _, _, torch = env
    g = torch.Generator(device="cuda").manual_seed(5)
    A = torch.randint(-127, 128, (520, 700), device="cuda", generator=g).float()
    B = torch.randint(-127, 128, (700, 390), device="cuda", generator=g).float()
    B[:, 0] = 0.0
    B[3, 0] = 4097.0
    C = product(env, A, B)
    assert np.array_equal(C, (A.double() @ B.double()).cpu().numpy().astype(np.float32))
    # a permutation of 24-bit values
    P = torch.eye(700, device="cuda")[torch.randperm(700, device="cuda", generator=g)]
    X = torch.randn(700, 390, device="cuda", generator=g)
    assert np.array_equal(product(env, P, X), (P.double() @ X.double()).cpu().numpy())


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e-30, 1e-42, 2.0 ** 55, 3e38])
@pytest.mark.parametrize("operand", [0, 1])
def test_operands_outside_the_range(env, value, operand):
    """One entry the pieces do not take (infinite, NaN, subnormal, extreme):
    the product is the CUDA cores', row and column of the entry included."""
    _, _, torch = env
    M, N, K = 300, 333, 400
    g = torch.Generator(device="cuda").manual_seed(9)
    A = torch.randn(M, K, device="cuda", generator=g)
    B = torch.randn(K, N, device="cuda", generator=g)
    (A if operand == 0 else B)[7, 5] = float(value)
    C = product(env, A, B)
    ref = (A.double() @ B.double()).cpu().numpy()
    fin = np.isfinite(ref) & (np.abs(ref) < 3.4e38)
    assert np.array_equal(np.isnan(C), np.isnan(ref))
    assert np.array_equal(C[~fin & ~np.isnan(ref)], ref[~fin & ~np.isnan(ref)].astype(np.float32))
    assert np.all(np.abs(C[fin] - ref[fin]) <= bound(A, B)[fin])
