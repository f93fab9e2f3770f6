"""The one-CTA tensor-core product in each of its tile widths (64, 128 and 256
columns, chosen by size), with remainders of the tile and of the 128-deep
stage, operands of odd leading dimension and 4-byte alignment, against the
binary64 product of the rounded operands; and the folded Freivalds check over
each width's column halves."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
PRODUCT = 3


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_6685_gb300 import safegpu as sg
    ctx = sg.sg_init(0, torch.cuda.current_stream().cuda_stream)
    yield sg, ctx, torch
    sg.sg_destroy(ctx)


# 64 columns, 128 columns (104 and 150 tiles for 152 SMs), 256 columns
SHAPES = [(1, 1, 1), (300, 200, 65), (129, 65, 129), (1000, 1000, 191), (1537, 1023, 193),
          (1280, 1920, 64), (2048, 2047, 65), (2049, 1800, 130)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("form", [0, 1])
def test_tile_widths(env, shape, prec, form):
    sg, ctx, torch = env
    M, N, K = shape
    g = torch.Generator(device="cuda").manual_seed(M + N + K)
    # a 4-byte offset: no 16-byte loads
    A = torch.randn(M * K + 1, device="cuda", generator=g)[1:].view(M, K)
    B = torch.randn(K, N, device="cuda", generator=g)
    ma, mb = sg.wrap_tensor(ctx, A), sg.wrap_tensor(ctx, B)
    sg.sg_sched_force(ctx, PRODUCT, form)
    try:
        mc = sg.sg_matmul(ctx, ma, mb, prec)
        C = sg.sg_matrix_read(ctx, mc, np.empty((M, N), np.float32))
    finally:
        sg.sg_sched_force(ctx, PRODUCT, -1)
    dt = torch.bfloat16 if prec == 1 else torch.float16
    a, b = A.to(dt).double(), B.to(dt).double()
    ref = (a @ b).cpu().numpy()
    # exact products, K / 16 truncating binary32 additions of sums of 16
    # (each at most 2 units of 2^-23)
    bound = ((a.abs() @ b.abs()) * ((K // 16 + 2) * 2.0 ** -22)).cpu().numpy()
    assert np.all(np.abs(C - ref) <= bound)
    for h in (mc, ma, mb):
        sg.sg_matrix_release(h)


@pytest.mark.parametrize("n", [200, 1000, 1400, 2100])
@pytest.mark.parametrize("form", [0, 1])
def test_folded_check_finds_a_planted_element(env, n, form):
    """An error planted in the first, a middle and the last column half."""
    sg, ctx, torch = env
    g = torch.Generator(device="cuda").manual_seed(n)
    A, B = (torch.randn(n, n, device="cuda", generator=g) for _ in range(2))
    ma, mb = sg.wrap_tensor(ctx, A), sg.wrap_tensor(ctx, B)
    sg.sg_sched_force(ctx, PRODUCT, form)
    try:
        for row, col in [(0, 0), (n // 2 + 1, n // 2 - 1), (n - 1, n - 1)]:
            sg.sg_debug_inject_matmul(ctx, row, col, 1e5)
            mc = sg.sg_matmul(ctx, ma, mb, sg.SG_PREC_BF16_TC)
            with pytest.raises(sg.SgError) as e:
                sg.sg_flush(ctx)
            assert e.value.status == sg.SG_ERR_POSTCONDITION
            assert sg.sg_last_violation(ctx).first_index == row
            sg.sg_matrix_release(mc)
        mc = sg.sg_matmul(ctx, ma, mb, sg.SG_PREC_BF16_TC)
        sg.sg_flush(ctx)
        sg.sg_matrix_release(mc)
    finally:
        sg.sg_sched_force(ctx, PRODUCT, -1)
