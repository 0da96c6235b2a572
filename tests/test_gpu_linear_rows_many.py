"""Linear row output with tuples that make many rows: the sizes around which they
are set aside, cut into pieces and dealt out, against the oracle; a capacity in the
middle of them; and the time they take beside the partitioned plan."""
import numpy as np
import pytest

import oracle
from paper_1905_13376_gb300 import binding

from gpu_util import cu, sorted_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


def lists(lens_r, lens_t, seed=0):
    """R with lens_r[b] tuples of every b, T with lens_t[c] of every c."""
    g = np.random.default_rng(seed)
    b = np.repeat(np.arange(len(lens_r)), lens_r).astype(np.int32)
    c = np.repeat(np.arange(len(lens_t)), lens_t).astype(np.int32)
    p, q = g.permutation(len(b)), g.permutation(len(c))
    return (g.integers(0, 1 << 20, len(b)).astype(np.int32), b[p]), (c[q], g.integers(0, 1 << 20, len(c)).astype(np.int32))


# rows per tuple: 127..129 (set aside above 128), 255..257 (pieces of 256), 1023..1025
# (spans of 1024), one list of a single entry on either side, many pieces
CASES = [([1], [127, 128, 129, 255, 256, 257]), ([127, 128, 129, 1023, 1024, 1025], [1]), ([31, 32, 33], [31, 32, 33]),
         ([5, 100, 700], [3, 90, 800]), ([3000], [1, 70])]


@pytest.mark.parametrize("lens", CASES)
@pytest.mark.parametrize("n", [1, 33, 700])
def test_rows_of_all_sizes(ctx, lens, n):
    R, T = lists(*lens)
    g = np.random.default_rng(n)
    S = (g.integers(0, len(lens[0]) + 1, n).astype(np.int32), g.integers(0, len(lens[1]) + 1, n).astype(np.int32))
    want = oracle.linear(R, S, T)["total"]
    if want > 6_000_000:
        S = (S[0][:20], S[1][:20])
        want = oracle.linear(R, S, T)["total"]
    rows = oracle.linear(R, S, T, oracle.MATERIALIZE, capacity=max(want, 1))["rows"]
    got = ctx.join3_linear(cu(R), cu(S), cu(T), "rows", capacity=want)
    assert int(got["n_rows"].item()) == want
    assert np.array_equal(sorted_rows(got["rows"].cpu().numpy()), rows[:want])


def test_capacity_among_the_tuples_set_aside(ctx):
    """Past the capacity nothing is written, and the number of rows is exact."""
    import ctypes
    import torch
    R, T = lists([40, 700, 3], [9, 500, 64])
    g = np.random.default_rng(3)
    S = (g.integers(0, 3, 400).astype(np.int32), g.integers(0, 3, 400).astype(np.int32))
    want = oracle.linear(R, S, T)["total"]
    have = {tuple(r) for r in oracle.linear(R, S, T, oracle.MATERIALIZE, capacity=want)["rows"].tolist()}
    d = [cu(x) for x in (R, S, T)]
    m = binding.MODES["rows"]
    for cap in (0, 1, 1000, want // 2, want - 1):
        o, res = ctx._outputs(m, None, cap + 4096, 4)
        o.capacity = cap
        res["rows"].fill_(-9)
        ws = ctx.workspace(ctx.workspace_size(binding.MWJ_LINEAR, *d, mode=m))
        hs = torch.cuda.current_stream().cuda_stream
        ctx._check(ctx.lib.mwj_join3_linear(ctx.h, *[binding._rel(x) for x in d], None, ctypes.byref(o), ws.data_ptr(),
                                            ws.numel(), hs))
        assert ctx.lib.mwj_stream_status(ctx.h, hs) == binding.MWJ_ERR_CAPACITY
        assert int(res["n_rows"].item()) == want
        assert bool((res["rows"][cap:] == -9).all()) and not bool((res["rows"][:cap] == -9).any())
        assert {tuple(r) for r in res["rows"][:cap].cpu().tolist()} <= have


@pytest.mark.parametrize("n,la,ld", [(64, 63, 64), (1024, 63, 64), (16384, 64, 80), (1024, 31, 32)])
def test_no_slower_than_the_partitioned_plan(ctx, n, la, ld):
    """Few tuples of many rows each: the default plan keeps up with the plan by
    H(B) buckets (it is four times faster or more; 1.25 leaves room for noise)."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    ri = lambda k, hi: torch.randint(0, hi, (k,), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
    key = torch.arange(64, device="cuda", dtype=torch.int32)
    R, T = (ri(64 * la, 1 << 20), key.repeat_interleave(la)), (key.repeat_interleave(ld), ri(64 * ld, 1 << 20))
    S = (ri(n, 64), ri(n, 64))
    sh = ctx.plan_shares(binding.MWJ_LINEAR, R, S, T, mode=binding.MODES["rows"])

    def time(shares):
        ts = []
        for k in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            ctx.join3_linear(R, S, T, "rows", shares=shares, capacity=n * la * ld, sync=False)
            e1.record()
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        return sorted(ts[2:])[2]

    assert time(None) < 1.25 * time(sh)
