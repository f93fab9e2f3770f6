"""The batched launch on a context whose stream is a caller's non-blocking
one, its first call queued behind work on the default stream: the lengths'
statistics (3000 collections on: by the device), the work list's counters and the
results are those of a context on the default stream."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_6685_gb300 import safegpu as sg
    return sg, torch


@pytest.mark.parametrize("nseg", [40, 2999, 3000, 12000])
def test_first_call_behind_the_default_stream(env, nseg):
    sg, torch = env
    r = np.random.default_rng(nseg)
    L = r.integers(0, 200, nseg)
    L[nseg // 3] = 70001
    off = np.concatenate([[0], np.cumsum(L)]).astype(np.int64)
    x = r.random(int(off[-1])).astype(np.float32)
    keep = x > 0.5
    kept = np.concatenate([[0], np.cumsum(keep)])
    c2 = np.concatenate([[0.0], np.cumsum(np.where(keep, x, 0).astype(np.float64))])
    want = c2[off[1:]] - c2[off[:-1]]
    # y = x * 1, pre x >= 0, keep x > 0.5
    ch = sg.chain([("x", 0), ("c", 1.0), ("mul",)], [("x", 0), ("c", 0.0), ("ge",)],
                  [("x", 0), ("c", 0.5), ("gt",)])
    to, tx = torch.from_numpy(off).cuda(), torch.from_numpy(x).cuda()
    bad = off.copy()
    bad[nseg // 2] = bad[nseg // 2 - 1] - 1
    tb = torch.from_numpy(bad).cuda()
    for _ in range(3):   # a new context each: its first call is the one
        s = torch.cuda.Stream()
        outs = (torch.empty(nseg, dtype=torch.float64, device="cuda"),
                torch.empty(nseg, dtype=torch.int64, device="cuda"),
                torch.empty(nseg, dtype=torch.int64, device="cuda"))
        ctx = sg.sg_init(0, s.cuda_stream)
        try:
            torch.cuda._sleep(2_000_000)
            s.wait_stream(torch.cuda.default_stream())
            for _ in range(2):
                sg.sg_batch_run(ctx, ch, tx.data_ptr(), to.data_ptr(), nseg,
                                *(t.data_ptr() for t in outs))
            with torch.cuda.stream(s):
                got = [t.cpu().numpy() for t in outs]
            with pytest.raises(sg.SgError) as e:
                sg.sg_batch_run(ctx, ch, tx.data_ptr(), tb.data_ptr(), nseg,
                                *(t.data_ptr() for t in outs))
            assert e.value.status == sg.SG_ERR_INVALID_ARG
        finally:
            sg.sg_destroy(ctx)
        assert np.array_equal(got[2], kept[off[1:]] - kept[off[:-1]])
        assert np.all(got[1] == -1)
        # at most 70001 values below 1 per collection, in pairs and by TwoSum: 2^-24
        # of each pair's sum; the reference's prefix sums 2^-53 of all
        assert np.all(np.abs(got[0] - want) <= 2.0 ** -23 * (want + 1) + len(x) ** 2 * 2.0 ** -53)
