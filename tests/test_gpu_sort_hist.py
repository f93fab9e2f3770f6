"""The sort around the size where its histogram changes form (2^22 keys): int32
and binary32, uniform, one-valued, from an address that is not a multiple of 16
bytes, checked and unchecked; bit for bit numpy's."""
import numpy as np
import pytest

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


@pytest.mark.parametrize("n", [(1 << 22) - 1, 1 << 22, (1 << 22) + 3, 5_000_001])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("kind", ["i32", "f32", "one", "off"])
def test_histogram_forms(env, n, shift, kind):
    sg, ctx, torch = env
    keys = inputs.sort_keys_uniform(n, seed=n)
    if kind == "one":
        keys[:] = -7
    if kind == "f32":   # finite, not zero: numpy's order is totalOrder
        f = keys.view(np.float32)
        keys = np.where(np.isfinite(f) & (f != 0), f, np.float32(1.5))
    t = torch.empty(n + shift, dtype=torch.float32 if kind == "f32" else torch.int32, device="cuda")
    t[shift:] = torch.from_numpy(keys).cuda()
    v = sg.sg_vector_wrap(ctx, sg.SG_F32 if kind == "f32" else sg.SG_I32, n,
                          t.data_ptr() + 4 * shift)
    if kind == "off":
        sg.sg_set_contract_mode(ctx, sg.SG_CONTRACTS_OFF)
    try:
        out = sg.sg_sort(ctx, v)
        got = sg.sg_vector_read(ctx, out, np.empty(n, keys.dtype))
    finally:
        sg.sg_set_contract_mode(ctx, sg.SG_CONTRACTS_PRE_POST)
    assert np.array_equal(got.view(np.uint32), np.sort(keys).view(np.uint32))
    sg.sg_vector_release(out)
    sg.sg_vector_release(v)
