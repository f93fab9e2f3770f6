"""Both forms of the elimination give the same bits.  A row-dominant matrix goes to
the one without interchanges.  Bordered by a row of ones, which is not
dominant but never a pivot row, and a column of zeros with a one below it, the same
matrix goes to the one with interchanges: its first pivots are the same, the last
is 1 and adds log 1 = 0, so that both determinants' logarithms are sums of the same
terms in the same order.  (Binary32 updates: sizes whose trailing blocks are all on
the tensor cores in either form; the form with interchanges takes the CUDA cores
for blocks of order 1537 to 1792.)"""
import numpy as np
import pytest

from paper_1410_6685_gb300 import inputs
from test_gpu_solve_diag import env   # noqa: F401

pytestmark = pytest.mark.gpu


def det(env, A, prec):   # noqa: F811
    sg, ctx, torch = env
    t = torch.from_numpy(np.ascontiguousarray(A, dtype=np.float32)).cuda()
    m = sg.wrap_tensor(ctx, t)
    sg.sg_det(ctx, m, prec)
    n0 = sg.sg_kernel_count(ctx)
    d = sg.sg_det(ctx, m, prec)
    n1 = sg.sg_kernel_count(ctx)
    sg.sg_matrix_release(m)
    return (d.sign, d.log_abs, d.info), n1 - n0


@pytest.mark.parametrize("n,prec", [(n, p) for n in (33, 127, 128, 129, 300, 385, 1000, 1600)
                                    for p in (0, 1, 2)] + [(2305, 1), (2305, 2)])
def test_same_bits(env, n, prec):   # noqa: F811
    A, _ = inputs.gepp_inputs(n)
    A[::3] *= -1.0
    B = np.zeros((n + 1, n + 1), np.float32)
    B[:n, :n] = A
    B[n] = 1.0
    without, k0 = det(env, A, prec)
    with_, k1 = det(env, B, prec)
    assert k0 < k1                     # the two forms
    assert without == with_
    assert without[2] == 0
