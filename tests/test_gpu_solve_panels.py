"""The elimination's panel forms by height (one CTA up to 256 rows, clusters of
8 and 16 beyond, two rows per thread above 4096) on general matrices, with
interchanges in every column, last panels narrower than 32, odd leading
dimensions, ties and a late zero pivot; against binary64 elimination with
partial pivoting."""
import numpy as np
import pytest

import oracle

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


@pytest.mark.parametrize("n", [33, 127, 255, 256, 257, 289, 300, 2047, 2081, 4129])
def test_heights(env, n):
    sg, ctx, torch = env
    g = torch.Generator(device="cuda").manual_seed(n)
    A = torch.randn(n, n, device="cuda", generator=g)
    xt = torch.randn(n, device="cuda", generator=g, dtype=torch.float64)
    b = A.double() @ xt
    ma, vb = sg.wrap_tensor(ctx, A), sg.wrap_tensor(ctx, b)
    opts = sg.SgSolveOpts()
    opts.precision = sg.SG_PREC_F32_SIMT
    x, info = sg.sg_solve(ctx, ma, vb, opts)
    got = sg.sg_vector_read(ctx, x, np.empty(n))
    ref = torch.linalg.solve(A.double(), b).cpu().numpy()
    assert np.max(np.abs(got - ref)) <= 1e-8 * max(1.0, np.max(np.abs(ref)))
    assert info.residual <= 1e-12
    # the portable panel does the same operations in the same order: the same
    # bits in every pivot
    d = sg.sg_det(ctx, ma)
    sg.sg_debug_portable_kernels(ctx, True)
    try:
        dp = sg.sg_det(ctx, ma)
    finally:
        sg.sg_debug_portable_kernels(ctx, False)
    assert d.info == 0 and (d.sign, d.log_abs) == (dp.sign, dp.log_abs)
    for h in (x, vb):
        sg.sg_vector_release(h)
    sg.sg_matrix_release(ma)


@pytest.mark.parametrize("n", [100, 300])
def test_ties_take_the_lowest_row(env, n):
    """Entries -1, 0, 1: most columns tie; the pivots' product is the oracle's."""
    sg, ctx, torch = env
    g = np.random.default_rng(n)
    A = g.integers(-1, 2, (n, n)).astype(np.float32)
    LU, piv, info = oracle.gepp_f64(A.astype(np.float64))
    assert info == 0 and np.any(piv != np.arange(n))
    u = np.diag(LU)
    sign = (-1) ** int(np.sum(piv != np.arange(n))) * int(np.prod(np.sign(u)))
    d = sg.sg_det(ctx, sg.wrap_tensor(ctx, torch.from_numpy(A).cuda()))
    assert d.info == 0 and d.sign == sign
    assert abs(d.log_abs - np.sum(np.log(np.abs(u)))) <= n * 2.0 ** -20


@pytest.mark.parametrize("n,k", [(200, 150), (400, 300), (2300, 2200)])
def test_late_zero_column(env, n, k):
    """A column of zeros makes step k's pivot exactly zero."""
    sg, ctx, torch = env
    A = np.random.default_rng(n).standard_normal((n, n)).astype(np.float32)
    A[:, k] = 0.0
    d = sg.sg_det(ctx, sg.wrap_tensor(ctx, torch.from_numpy(A).cuda()))
    assert d.sign == 0 and d.info == k + 1 and d.det == 0.0
