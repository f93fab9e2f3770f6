"""A binary32 product's scratch, its operands' pieces (6 bytes an entry): bounded
after the product is done, given back with the context."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_6685_gb300 import safegpu as sg
    return sg, torch


def free(torch):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def rows(A, B, C, k):
    """The largest error of k rows of C against binary64, relative to sum |a b|."""
    i = np.linspace(0, A.shape[0] - 1, k).astype(int)
    a = A[i].double()
    ref, mag = a @ B.double(), a.abs() @ B.double().abs()
    return float(((C[i].double() - ref) / mag).abs().max())


def test_large_products_give_their_scratch_back(env):
    """Two products of 1.9 and 0.3 GB of pieces: a GB may stay, and the small
    product's block (64 MB), beside the results' pool; all goes with the context."""
    sg, torch = env
    A, B = torch.randn(20000, 8000, device="cuda"), torch.randn(8000, 20000, device="cuda")
    a2, b2 = A[:5000, :5000].contiguous(), B[:5000, :5000].contiguous()
    before = free(torch)
    ctx = sg.sg_init(0, torch.cuda.current_stream().cuda_stream)
    warm = free(torch)
    results = 0
    for x, y in ((A, B), (a2, b2), (a2, b2)):
        ma, mb = sg.wrap_tensor(ctx, x), sg.wrap_tensor(ctx, y)
        mc = sg.sg_matmul(ctx, ma, mb, sg.SG_PREC_F32_SIMT)
        C = torch.from_numpy(sg.sg_matrix_read(ctx, mc, np.empty((x.shape[0], y.shape[1]), np.float32)))
        K = x.shape[1]
        assert rows(x, y, C.cuda(), 7) <= (24 + K / 16) * 2.0 ** -24
        del C
        torch.cuda.empty_cache()
        results += x.shape[0] * y.shape[1] * 4
        for h in (mc, ma, mb):
            sg.sg_matrix_release(h)
        # (32 MB granules, and the check's scratch)
        assert warm - free(torch) <= results + 1024 * MB + 64 * MB + 192 * MB
    sg.sg_destroy(ctx)
    assert before - free(torch) <= results + 192 * MB


def test_repeated_small_products_share_a_block(env):
    sg, torch = env
    ctx = sg.sg_init(0, torch.cuda.current_stream().cuda_stream)
    try:
        for n in (300, 1000, 700, 1300, 300):
            A = torch.randn(n, n, device="cuda")
            B = torch.randn(n, n, device="cuda")
            ma, mb = sg.wrap_tensor(ctx, A), sg.wrap_tensor(ctx, B)
            cs = [sg.sg_matmul(ctx, ma, mb, sg.SG_PREC_F32_SIMT) for _ in range(3)]
            for mc in cs:
                C = sg.sg_matrix_read(ctx, mc, np.empty((n, n), np.float32))
                assert rows(A, B, torch.from_numpy(C).cuda(), 20) <= (24 + n / 16) * 2.0 ** -24
            for h in cs + [ma, mb]:
                sg.sg_matrix_release(h)
    finally:
        sg.sg_destroy(ctx)
