"""Elimination without interchanges whose next diagonal block runs beside the
trailing update (16-bit updates): sizes where the update leaves out its first
128 x 128 entries in a lone tile, a ragged one or a wave of them, in the CTA-pair
and the one-CTA form, and a verification that fails while an update is in
flight.  Tolerances as for the other dominant matrices: refinement reaches 1e-9
of the oracle's solution, the determinant 2^-12 per pivot."""
import numpy as np
import pytest

from paper_1410_6685_gb300 import inputs
from test_gpu_solve_diag import check, env   # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("portable", [False, True])
@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("n", [256, 258, 383, 384, 513, 1100, 2305])
def test_corner_left_out(env, n, prec, portable):   # noqa: F811
    sg, ctx, _ = env
    A, _ = inputs.gepp_inputs(n)
    A[1::3] *= -1.0
    sg.sg_debug_portable_kernels(ctx, portable)
    try:
        check(env, A, prec)
    finally:
        sg.sg_debug_portable_kernels(ctx, False)


@pytest.mark.parametrize("prec", [1])   # these entries are past fp16's range
@pytest.mark.parametrize("n,swap", [(400, 130), (900, 260), (1500, 128)])
def test_verification_fails_beside_an_update(env, n, swap, prec):   # noqa: F811
    """Rows from `swap` on outgrow earlier pivots (still dominant): the diagonal
    block that finds out runs beside an update that must not see its report."""
    A, _ = inputs.gepp_inputs(n)
    A[swap:, :swap] = 0.0
    off = np.abs(A.astype(np.float64)).sum(axis=1) - np.abs(np.diag(A).astype(np.float64))
    A[np.arange(n), np.arange(n)] = (off * 1.01 + 1.0).astype(np.float32)
    A[swap:] *= (2.0 ** (3 * (np.arange(n - swap) % 5)))[:, None].astype(np.float32)
    check(env, A, prec)
