"""Fused stream passes at the lengths where a thread takes one or two vectors
of four at a time and where the launch has one or several waves of CTAs: every
element computed, the first violation found wherever it stands, and the sum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ADD = [("x", 0), ("x", 1), ("add",)]


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_6685_gb300 import safegpu as sg
    ctx = sg.sg_init(0, torch.cuda.current_stream().cuda_stream)
    yield sg, ctx, torch
    sg.sg_destroy(ctx)


def lengths():
    """Around one, two and 64 steps of the largest grid (8 CTAs of 256 threads
    per SM, four elements a thread); a GB300 has 152 SMs."""
    step = 152 * 8 * 256 * 4
    return [1, 5, 1023, 1024, 1027, step - 1, step, step + 1, step + 1029, 2 * step + 3,
            3 * step - 4, 16 * step + 7, 64 * step + 1025]


@pytest.mark.parametrize("n", lengths())
def test_elements_sum_and_first_violation(env, n):
    sg, ctx, torch = env
    g = torch.Generator(device="cuda").manual_seed(n)
    x, y = (torch.rand(n, device="cuda", generator=g) * 2 - 1 for _ in range(2))
    vx, vy = sg.wrap_tensor(ctx, x), sg.wrap_tensor(ctx, y)
    z = sg.sg_zip(ctx, ADD, vx, vy)
    s = sg.sg_reduce(ctx, sg.SG_REDUCE_SUM, z)
    total = sg.sg_scalar_get(ctx, s)
    got = sg.sg_vector_read(ctx, z, np.empty(n, np.float32))
    want = x + y
    assert np.array_equal(got, want.cpu().numpy())
    # per thread k values of magnitude <= 2 by TwoSum, whose k error terms (each
    # at most 2^-24 of a partial sum <= 2k) are added in binary32; the threads'
    # sums in binary64, by at most 64 additions each
    k = n / (152 * 8 * 256) + 8
    assert abs(total - float(want.double().sum())) <= n * 2 * k * k * 2.0 ** -48 + 2 * n * 64 * 2.0 ** -53
    sg.sg_vector_release(z)
    sg.sg_scalar_release(s)
    # z <= 2 holds but for one planted element, with another behind it
    limit = sg.contract(sg.SG_C_FOR_ALL, [("x", 0), ("c", 2.0), ("le",)])
    for i in sorted({0, n // 3, n // 2 + 513, n - 2, n - 1}):
        if not 0 <= i < n:
            continue
        keep = x[i].item(), x[n - 1].item()
        x[n - 1] = 6.0
        x[i] = 5.0
        z = sg.sg_zip(ctx, ADD, vx, vy)
        sg.sg_ensure(ctx, z, limit)
        with pytest.raises(sg.SgError) as e:
            sg.sg_flush(ctx)
        assert e.value.status == sg.SG_ERR_POSTCONDITION
        assert sg.sg_last_violation(ctx).first_index == i
        sg.sg_vector_release(z)
        x[n - 1] = keep[1]
        x[i] = keep[0]
    for h in (vx, vy):
        sg.sg_vector_release(h)
