"""Small eliminations take the form that is shorter for them: up to one panel (32
rows) the one with interchanges at once, up to 256 rows the one without only where
no entry below the diagonal is larger than it.  Seen from the number of kernels a
determinant launches; the results are the oracle's either way."""
import numpy as np
import pytest

from paper_1410_6685_gb300 import inputs
from test_gpu_solve_diag import check, env   # noqa: F401

pytestmark = pytest.mark.gpu


def outgrown(n):
    """Row-dominant, but rows scaled so that their entries outgrow the pivots above."""
    A, _ = inputs.gepp_inputs(n)
    off = np.abs(A.astype(np.float64)).sum(axis=1) - np.abs(np.diag(A).astype(np.float64))
    A[np.arange(n), np.arange(n)] = (off * 1.01 + 1.0).astype(np.float32)
    return A * (2.0 ** (3 * (np.arange(n) % 5)))[:, None].astype(np.float32)


def launches(env, A, prec):   # noqa: F811
    sg, ctx, torch = env
    t = torch.from_numpy(np.ascontiguousarray(A, dtype=np.float32)).cuda()
    m = sg.wrap_tensor(ctx, t)
    sg.sg_det(ctx, m, prec)          # (workspace and graph)
    n0 = sg.sg_kernel_count(ctx)
    sg.sg_det(ctx, m, prec)
    n1 = sg.sg_kernel_count(ctx)
    sg.sg_matrix_release(m)
    return n1 - n0


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", [2, 31, 32, 33, 100, 128, 129, 255, 256])
def test_one_elimination(env, n, prec):   # noqa: F811
    general = launches(env, np.random.default_rng(n).standard_normal((n, n)), prec)
    assert launches(env, outgrown(n), prec) == general
    check(env, outgrown(n), prec)
    A, _ = inputs.gepp_inputs(n)
    if n <= 32:
        assert launches(env, A, prec) == general
    else:
        assert launches(env, A, prec) < general
    check(env, A, prec)


def test_larger_matrices_are_verified(env):   # noqa: F811
    """Above 256 rows the columns are not looked at: the form without interchanges
    is tried, and the one with them follows."""
    n = 257
    general = launches(env, np.random.default_rng(n).standard_normal((n, n)), 0)
    assert launches(env, outgrown(n), 0) > general
    check(env, outgrown(n), 0)
