"""A trailing update of the elimination that gives up a wait: its report (the
host raises the word that the update's kernels raise) ends sg_solve and sg_det
with SG_ERR_TIMEOUT in every precision, never with a result, and the context
then gives the oracle's results again."""
import numpy as np
import pytest

from paper_1410_6685_gb300 import inputs
from test_gpu_solve_diag import check, env, solve   # noqa: F401

pytestmark = pytest.mark.gpu


def attempt(env, A, prec, what):   # noqa: F811
    sg, ctx, torch = env
    ta = torch.from_numpy(A.astype(np.float32)).cuda()
    ma = sg.wrap_tensor(ctx, ta)
    try:
        if what == "det":
            return sg.sg_det(ctx, ma, prec)
        tb = torch.from_numpy(A.astype(np.float64).sum(axis=1)).cuda()
        vb = sg.wrap_tensor(ctx, tb)
        opts = sg.SgSolveOpts()
        opts.precision = prec
        try:
            x, _ = sg.sg_solve(ctx, ma, vb, opts)
            sg.sg_vector_release(x)
        finally:
            sg.sg_vector_release(vb)
    finally:
        sg.sg_matrix_release(ma)


@pytest.mark.parametrize("what", ["det", "solve"])
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("n", [300, 1100])
def test_update_wait_gave_up(env, n, prec, what):   # noqa: F811
    sg, ctx, _ = env
    A = np.random.default_rng(n).standard_normal((n, n))
    sg.sg_debug_inject_update_timeout(ctx)
    with pytest.raises(sg.SgError) as e:
        attempt(env, A, prec, what)
    assert e.value.status == sg.SG_ERR_TIMEOUT
    if prec == 0:
        check(env, A, prec, tol=1e-8)
    else:
        attempt(env, A, prec, "det")


def test_switch(env):   # noqa: F811
    """Switched off again, nothing is reported; an elimination without
    interchanges leaves the switch for the next one with them."""
    sg, ctx, _ = env
    A = np.random.default_rng(1).standard_normal((200, 200))
    sg.sg_debug_inject_update_timeout(ctx, True)
    sg.sg_debug_inject_update_timeout(ctx, False)
    attempt(env, A, 0, "det")
    sg.sg_debug_inject_update_timeout(ctx, True)
    attempt(env, inputs.gepp_inputs(300)[0], 1, "det")
    with pytest.raises(sg.SgError):
        attempt(env, A, 0, "det")
    with pytest.raises(sg.SgError):
        sg.sg_debug_inject_update_timeout(None)
