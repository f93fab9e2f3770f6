"""Elimination without interchanges (diagonally dominant matrices) and its
fallback to the general form, through the C ABI against the binary64 oracle:
the edges of its 128-column blocks, 64-wide border strips and update operands
in every precision, matrices that pass the dominance screen but do need
interchanges, and entries outside the split operands' range."""
import numpy as np
import pytest

import oracle
from paper_1410_6685_gb300 import inputs

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


def solve(env, A, b, prec):
    sg, ctx, torch = env
    ta = torch.from_numpy(np.ascontiguousarray(A, dtype=np.float32)).cuda()
    tb = torch.from_numpy(np.ascontiguousarray(b, dtype=np.float64)).cuda()
    ma, vb = sg.wrap_tensor(ctx, ta), sg.wrap_tensor(ctx, tb)
    opts = sg.SgSolveOpts()
    opts.precision = prec
    x, info = sg.sg_solve(ctx, ma, vb, opts)
    xs = sg.sg_vector_read(ctx, x, np.empty(len(b), np.float64))
    d = sg.sg_det(ctx, ma, prec)
    for h in (x, vb):
        sg.sg_vector_release(h)
    sg.sg_matrix_release(ma)
    return xs, info, d


def check(env, A, prec, tol=1e-9):
    n = len(A)
    A = A.astype(np.float32)
    xt = np.random.default_rng(n).standard_normal(n)
    b = A.astype(np.float64) @ xt
    x, info, d = solve(env, A, b, prec)
    ref = oracle.solve(A, b)
    assert np.max(np.abs(x - ref)) <= tol * max(1.0, np.max(np.abs(ref)))
    assert info.residual <= 1e-12 and info.info == 0
    LU, piv, _ = oracle.gepp_f64(A.astype(np.float64))
    u = np.diag(LU)
    sign = (-1) ** int(np.sum(piv != np.arange(n))) * int(np.prod(np.sign(u)))
    assert d.sign == sign and d.info == 0
    # per pivot, as for the other determinants: 2^-20 binary32, 2^-12 bf16
    assert abs(d.log_abs - np.sum(np.log(np.abs(u)))) <= n * 2.0 ** (-20 if prec == 0 else -12)


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 191, 193, 257, 385, 1000])
def test_dominant_edges(env, n, prec):
    A, _ = inputs.gepp_inputs(n)
    A[::3] *= -1.0    # negative pivots too
    check(env, A, prec)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n,swap", [(100, 0), (300, 0), (300, 200), (700, 500)])
def test_dominant_rows_that_need_interchanges(env, n, swap, prec):
    """Rows scaled by powers of two from row `swap` on stay dominant, but
    their entries outgrow earlier pivots: the verification fails at that block
    and the general elimination gives the oracle's pivots."""
    A, _ = inputs.gepp_inputs(n)
    A[swap:, :swap] = 0.0     # the pivots before `swap` stay on the diagonal
    off = np.abs(A.astype(np.float64)).sum(axis=1) - np.abs(np.diag(A).astype(np.float64))
    A[np.arange(n), np.arange(n)] = (off * 1.01 + 1.0).astype(np.float32)
    # dominance is kept, just
    A[swap:] *= (2.0 ** (3 * (np.arange(n - swap) % 5)))[:, None].astype(np.float32)
    LU, piv, _ = oracle.gepp_f64(A.astype(np.float64))
    assert np.flatnonzero(piv != np.arange(n))[0] >= swap
    check(env, A, prec)


def test_zero_pivot_under_the_screen(env):
    """A zero row passes 2 |a_ii| >= sum |a_ij|: the general form reports it."""
    sg, ctx, torch = env
    A, b = inputs.gepp_inputs(200)
    A[150] = 0.0
    ta, tb = torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda()
    with pytest.raises(sg.SgError) as e:
        sg.sg_solve(ctx, sg.wrap_tensor(ctx, ta), sg.wrap_tensor(ctx, tb))
    assert e.value.status == sg.SG_ERR_SINGULAR


@pytest.mark.parametrize("scale", [2.0 ** -70, 2.0 ** 60])
def test_dominant_outside_the_pieces_range(env, scale):
    """Binary32 updates of a matrix whose entries the three bf16 pieces do not
    take: the CUDA cores' update, the same solution."""
    A, _ = inputs.gepp_inputs(300)
    check(env, A * np.float32(scale), 0)


def test_general_after_dominant_in_one_context(env):
    """Both factorisation graphs of one size, in turn."""
    g = np.random.default_rng(3)
    n = 260
    for _ in range(2):
        check(env, inputs.gepp_inputs(n)[0], 0)
        check(env, g.standard_normal((n, n)), 0, tol=1e-8)
