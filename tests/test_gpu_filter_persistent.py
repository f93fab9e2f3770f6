"""The persistent filter (8192-item tiles, positions from one scanning warp)
where its CTAs take several tiles each: sizes around one and two rounds of
the resident CTAs, everything and nothing kept, an unaligned input, a folded
postcondition in a late tile, and a late tile that never publishes."""
import time

import numpy as np
import pytest

import oracle
from paper_1410_6685_gb300 import inputs

pytestmark = pytest.mark.gpu
FILTER, TILE = 2, 8192


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_6685_gb300 import safegpu as sg
    ctx = sg.sg_init(0, torch.cuda.current_stream().cuda_stream)
    sg.sg_sched_force(ctx, FILTER, 2)
    yield sg, ctx, torch
    sg.sg_debug_lookback(ctx, 0, -1)
    sg.sg_destroy(ctx)


def kept(env, t, pred, post=None):
    sg, ctx, _ = env
    v = sg.sg_vector_wrap(ctx, sg.SG_F32, t.numel(), t.data_ptr())
    k = sg.sg_filter(ctx, pred, v)
    if post is not None:
        sg.sg_ensure(ctx, k, sg.contract(sg.SG_C_FOR_ALL, post))
    try:
        sg.sg_flush(ctx)
        m = sg.sg_vector_count(ctx, k)
        return sg.sg_vector_read(ctx, k, np.empty(m, np.float32)) if m else np.empty(0, np.float32)
    finally:
        sg.sg_vector_release(k)
        sg.sg_vector_release(v)


# 607 CTAs take tiles: one round, a tile more, two rounds and a part of a tile
@pytest.mark.parametrize("n", [607 * TILE, 608 * TILE, 1215 * TILE + 77])
@pytest.mark.parametrize("above", [-2.0, 0.25, 2.0])
@pytest.mark.parametrize("offset", [0, 1])
def test_rounds(env, n, above, offset):
    _, _, torch = env
    x = inputs.uniform_pm1(inputs.rng(n), n + offset)
    t = torch.from_numpy(x).cuda()[offset:]
    pred = [("x", 0), ("c", above), ("gt",)]
    got = kept(env, t, pred)
    assert np.array_equal(got.view(np.uint32), oracle.filter(pred, x[offset:]).view(np.uint32))


def test_postcondition_in_a_late_tile(env):
    sg, ctx, torch = env
    n = 1300 * TILE + 5
    x = inputs.uniform_pm1(inputs.rng(4), n)
    x[n - 3] = 0.9999999
    x[n - 9000] = 0.9999999
    pred = [("x", 0), ("c", 0.0), ("gt",)]
    post = [("x", 0), ("c", 0.99999985), ("lt",)]
    keep = oracle.filter(pred, x)
    first = int(np.flatnonzero(~(keep < np.float32(0.99999985)))[0])
    with pytest.raises(sg.SgError) as e:
        kept(env, torch.from_numpy(x).cuda(), pred, post)
    assert e.value.status == sg.SG_ERR_POSTCONDITION
    assert sg.sg_last_violation(ctx).first_index == first


@pytest.mark.parametrize("skip", [0, 606, 700, 1290])
def test_late_tile_that_never_publishes(env, skip):
    sg, ctx, torch = env
    n = 1300 * TILE
    x = inputs.uniform_pm1(inputs.rng(5), n)
    t = torch.from_numpy(x).cuda()
    pred = [("x", 0), ("c", 0.25), ("gt",)]
    sg.sg_debug_lookback(ctx, 2000, skip)
    t0 = time.time()
    try:
        with pytest.raises(sg.SgError) as e:
            kept(env, t, pred)
    finally:
        sg.sg_debug_lookback(ctx, 0, -1)
    assert e.value.status == sg.SG_ERR_TIMEOUT
    assert time.time() - t0 < 10.0
    got = kept(env, t, pred)
    assert np.array_equal(got.view(np.uint32), oracle.filter(pred, x).view(np.uint32))
