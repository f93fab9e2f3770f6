"""The batched launch around the counts where its set-up changes form (3000
collections: their lengths' statistics by the device; more than 1024: several
collections per thread of the work list's scan): every collection's sum, count
and first violation, empty collections among them, and refused offsets."""
import numpy as np
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


def setup(env, L, seed):
    sg, ctx, torch = env
    off = np.concatenate([[0], np.cumsum(L)]).astype(np.int64)
    x = np.random.default_rng(seed).random(int(off[-1])).astype(np.float32)
    to, tx = torch.from_numpy(off).cuda(), torch.from_numpy(x).cuda()
    n = len(L)
    outs = (torch.empty(n, dtype=torch.float64, device="cuda"),
            torch.empty(n, dtype=torch.int64, device="cuda"),
            torch.empty(n, dtype=torch.int64, device="cuda"))
    # y = x * 1, pre x >= 0, keep x > 0.5
    ch = sg.chain([("x", 0), ("c", 1.0), ("mul",)], [("x", 0), ("c", 0.0), ("ge",)],
                  [("x", 0), ("c", 0.5), ("gt",)])
    return off, x, to, tx, outs, ch


@pytest.mark.parametrize("nseg", [1, 1023, 1025, 2999, 3000, 3001, 5000, 40000])
def test_counts(env, nseg):
    sg, ctx, torch = env
    r = np.random.default_rng(nseg)
    L = r.integers(0, 60, nseg)
    L[nseg // 2] = 20001          # several chunks of any schedule but the longest
    off, x, to, tx, outs, ch = setup(env, L, nseg)
    sg.sg_batch_run(ctx, ch, tx.data_ptr(), to.data_ptr(), nseg, *(t.data_ptr() for t in outs))
    keep = x > 0.5
    c1 = np.concatenate([[0], np.cumsum(keep)])
    assert np.array_equal(outs[2].cpu().numpy(), c1[off[1:]] - c1[off[:-1]])
    assert np.all(outs[1].cpu().numpy() == -1)
    c2 = np.concatenate([[0.0], np.cumsum(np.where(keep, x, 0).astype(np.float64))])
    want = c2[off[1:]] - c2[off[:-1]]
    # at most 20001 values below 1 per collection, in pairs and by TwoSum: 2^-24 of
    # each pair's sum; the reference's prefix sums 2^-53 of all
    assert np.all(np.abs(outs[0].cpu().numpy() - want) <= 2.0 ** -23 * (want + 1) + len(x) ** 2 * 2.0 ** -53)


@pytest.mark.parametrize("nseg", [2999, 3000, 10000])
def test_decreasing_offsets_are_refused(env, nseg):
    sg, ctx, torch = env
    off, x, to, tx, outs, ch = setup(env, np.full(nseg, 5), 1)
    for i in (1, nseg // 2, nseg):
        bad = off.copy()
        bad[i] = bad[i - 1] - 1
        tb = torch.from_numpy(bad).cuda()
        with pytest.raises(sg.SgError) as e:
            sg.sg_batch_run(ctx, ch, tx.data_ptr(), tb.data_ptr(), nseg,
                            *(t.data_ptr() for t in outs))
        assert e.value.status == sg.SG_ERR_INVALID_ARG
