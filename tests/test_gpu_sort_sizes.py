"""The sort around the sizes where its tile changes (2048, 4096 and 6144 keys)
and around whole tiles of the smaller two, int32 and binary32 keys, uniform,
few-valued and descending, with its postconditions; bit for bit numpy's."""
import numpy as np
import pytest

from paper_1410_6685_gb300 import inputs

pytestmark = pytest.mark.gpu

SIZES = [2047, 2048, 2049, 17 * 2048, 199_999, 200_000, 200_001, 60 * 4096 - 1, 60 * 4096,
         60 * 4096 + 1, 1_999_999, 2_000_001]


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_6685_gb300 import safegpu as sg
    ctx = sg.sg_init(0, torch.cuda.current_stream().cuda_stream)
    yield sg, ctx, torch
    sg.sg_destroy(ctx)


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("kind", ["uniform", "few", "descending"])
@pytest.mark.parametrize("dt", ["i32", "f32"])
def test_sizes(env, n, kind, dt):
    sg, ctx, torch = env
    keys = inputs.sort_keys_uniform(n, seed=n)
    if kind == "few":
        keys = inputs.sort_keys_distinct(n, 5)
    elif kind == "descending":
        keys = np.sort(keys)[::-1].copy()
    if dt == "f32":   # finite values: numpy's order is totalOrder
        keys = np.where(np.isfinite(keys.view(np.float32)), keys.view(np.float32),
                        np.float32(1.5))
        keys = np.where(keys == 0, np.float32(2.5), keys)
    t = torch.from_numpy(keys).cuda()
    v = sg.sg_vector_wrap(ctx, sg.SG_I32 if dt == "i32" else sg.SG_F32, n, t.data_ptr())
    out = sg.sg_sort(ctx, v)
    sg.sg_flush(ctx)
    got = sg.sg_vector_read(ctx, out, np.empty(n, keys.dtype))
    assert np.array_equal(got.view(np.uint32), np.sort(keys).view(np.uint32))
    sg.sg_vector_release(out)
    sg.sg_vector_release(v)


@pytest.mark.parametrize("n", [50_000, 500_000])
def test_contracts_off(env, n):
    sg, ctx, torch = env
    keys = inputs.sort_keys_uniform(n, seed=n)
    t = torch.from_numpy(keys).cuda()
    v = sg.sg_vector_wrap(ctx, sg.SG_I32, n, t.data_ptr())
    sg.sg_set_contract_mode(ctx, sg.SG_CONTRACTS_OFF)
    try:
        out = sg.sg_sort(ctx, v)
        got = sg.sg_vector_read(ctx, out, np.empty(n, np.int32))
    finally:
        sg.sg_set_contract_mode(ctx, sg.SG_CONTRACTS_PRE_POST)
    assert np.array_equal(got, np.sort(keys))
