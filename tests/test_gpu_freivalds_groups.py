"""The product's randomised check at the sizes where its passes change how many
rows or columns a CTA takes: an error planted in the first, a middle and the last
row is found there, and the clean product passes.  1e5 in one element is above
the check's bound at every size here: with 8 u sqrt(sum a^2 ((B r)^2 + |B|^2)),
u <= 2^-8 and entries of variance 1, the root is about sqrt(2) n < 4300."""
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


NS = [9, 65, 500, 830, 1000, 1215, 1218, 1700, 2431, 3000]


def places(n):
    return [(0, 0), (n // 2 + 1, n // 2 - 1), (n - 1, n - 1)]


def violation(sg, ctx):
    with pytest.raises(sg.SgError) as e:
        sg.sg_flush(ctx)
    assert e.value.status == sg.SG_ERR_POSTCONDITION
    return sg.sg_last_violation(ctx).first_index


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("n", NS)
def test_folded_check(env, n, prec):
    """The check folded into a tensor-core product, the error planted in it."""
    sg, ctx, torch = env
    g = torch.Generator(device="cuda").manual_seed(n)
    A, B = (torch.randn(n, n, device="cuda", generator=g) for _ in range(2))
    ma, mb = sg.wrap_tensor(ctx, A), sg.wrap_tensor(ctx, B)
    for row, col in places(n):
        sg.sg_debug_inject_matmul(ctx, row, col, 1e5)
        mc = sg.sg_matmul(ctx, ma, mb, prec)
        assert violation(sg, ctx) == row
        sg.sg_matrix_release(mc)
    mc = sg.sg_matmul(ctx, ma, mb, prec)
    sg.sg_flush(ctx)
    for h in (mc, ma, mb):
        sg.sg_matrix_release(h)


@pytest.mark.parametrize("n", NS)
def test_separate_check(env, n):
    """The check as passes of its own: ensured by the caller on a given matrix,
    and the binary32 product's own."""
    sg, ctx, torch = env
    g = torch.Generator(device="cuda").manual_seed(n)
    A, B = (torch.randn(n, n, device="cuda", generator=g) for _ in range(2))
    ma, mb = sg.wrap_tensor(ctx, A), sg.wrap_tensor(ctx, B)
    check = sg.contract(sg.SG_C_FREIVALDS, other=[ma, mb], seed=6, nvec=4, tol=8.0)
    C = (A.double() @ B.double()).float()
    for row, col in places(n) + [(None, None)]:
        D = C.clone()
        if row is not None:
            D[row, col] += 1e5
        md = sg.wrap_tensor(ctx, D)
        sg.sg_ensure(ctx, md, check)
        if row is not None:
            assert violation(sg, ctx) == row
        else:
            sg.sg_flush(ctx)
        sg.sg_matrix_release(md)
    mc = sg.sg_matmul(ctx, ma, mb, 0)
    sg.sg_flush(ctx)
    for h in (mc, ma, mb):
        sg.sg_matrix_release(h)
