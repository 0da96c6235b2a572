"""Row output of the linear join without shares (lists of R and T, S streamed):
ragged chunks, tuples with no, few and very many rows, both layouts of either
list, key -1, empty relations, capacity, and the partitioned plan on the same
inputs.  Rows compared after sorting."""
import numpy as np
import pytest

import oracle
from paper_1905_13376_gb300 import binding

from gpu_util import cu, sorted_rows

pytestmark = pytest.mark.gpu

DENSE = lambda k: (k - 3).astype(np.int32)
SPREAD = lambda k: ((k * 2654435761 + 12345) % (1 << 32) - (1 << 31)).astype(np.int32)
MARK = lambda k: np.where(k % 4 == 0, -1, (1 << 31) - 1 - k).astype(np.int32)


@pytest.fixture(scope="module")
def ctx():
    import torch
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


def check(ctx, R, S, T, shares=(None,)):
    n = oracle.linear(R, S, T, oracle.COUNT)["total"]
    want = oracle.linear(R, S, T, oracle.MATERIALIZE, capacity=n)["rows"]
    for sh in shares:
        got = ctx.join3_linear(cu(R), cu(S), cu(T), "rows", shares=sh, capacity=n + 3)
        assert int(got["n_rows"].item()) == n and int(got["total"].item()) == n
        assert np.array_equal(sorted_rows(got["rows"].cpu().numpy()), want)
    return n


@pytest.mark.parametrize("fb", [DENSE, SPREAD, MARK])
@pytest.mark.parametrize("fc", [DENSE, SPREAD, MARK])
@pytest.mark.parametrize("n", [1, 33, 511, 513, 5000])
def test_layouts_and_chunks(ctx, fb, fc, n):
    g = np.random.default_rng(n)
    dom = max(2, n // 2)
    R = (g.integers(-5, 90, n + 1).astype(np.int32), fb(g.integers(0, dom, n + 1)))
    S = (fb(g.integers(0, dom, n)), fc(g.integers(0, dom, n)))
    T = (fc(g.integers(0, dom, n + 2)), g.integers(-1000, 1000, n + 2).astype(np.int32))
    if n == 5000 and (fb is MARK or fc is MARK):
        S = (S[0][:200], S[1][:200])   # (a quarter of the keys is one key)
        R = (R[0][:900], R[1][:900])
        T = (T[0][:900], T[1][:900])
    check(ctx, R, S, T, shares=(None, (16, 1, 1)))


@pytest.mark.parametrize("nr,nt", [(64, 64), (4096, 1), (4097, 1), (1, 4097), (300, 900)])
def test_tuples_with_many_rows(ctx, nr, nt):
    """One (b, c) whose rows are at, just above and far above what a warp writes
    itself, beside tuples with few and none."""
    g = np.random.default_rng(nr + nt)
    R = (g.integers(0, 9999, nr + 50).astype(np.int32), np.r_[np.full(nr, 7), g.integers(100, 150, 50)].astype(np.int32))
    T = (np.r_[np.full(nt, 3), g.integers(200, 240, 50)].astype(np.int32), g.integers(0, 9999, nt + 50).astype(np.int32))
    S = (np.r_[g.integers(100, 160, 700), 7, 7].astype(np.int32), np.r_[g.integers(200, 250, 700), 3, 3].astype(np.int32))
    assert check(ctx, R, S, T) >= 2 * nr * nt


def test_empty_and_capacity(ctx):
    E = (np.zeros(0, np.int32), np.zeros(0, np.int32))
    g = np.random.default_rng(3)
    rel = lambda n: (g.integers(0, 12, n).astype(np.int32), g.integers(0, 12, n).astype(np.int32))
    R, S, T = rel(100), rel(100), rel(100)
    for args in ((E, S, T), (R, E, T), (R, S, E), (E, E, E)):
        got = ctx.join3_linear(*[cu(x) for x in args], "rows", capacity=5)
        assert int(got["n_rows"].item()) == 0 and int(got["total"].item()) == 0
    n = oracle.linear(R, S, T, oracle.COUNT)["total"]
    with pytest.raises(binding.MwjError) as e:
        ctx.join3_linear(cu(R), cu(S), cu(T), "rows", capacity=n - 1)
    assert e.value.status == binding.MWJ_ERR_CAPACITY
    check(ctx, R, S, T)


@pytest.mark.parametrize("nr,nt,short", [(3, 5, 1), (4097, 1, 1), (4097, 1, 4000), (300, 900, 500_000)])
def test_rows_past_the_capacity(ctx, nr, nt, short):
    """They are counted and not written, also in the middle of a tuple with many rows."""
    import ctypes
    import torch
    R = (np.arange(nr, dtype=np.int32), np.full(nr, 7, np.int32))
    T = (np.full(nt, 3, np.int32), np.arange(nt, dtype=np.int32))
    S = (np.full(2, 7, np.int32), np.full(2, 3, np.int32))
    n = 2 * nr * nt
    dR, dS, dT = cu(R), cu(S), cu(T)
    m = binding.MODES["rows"]
    o, res = ctx._outputs(m, None, n, 4)
    res["rows"].fill_(-7)
    o.capacity = n - short
    ws = ctx.workspace(ctx.workspace_size(binding.MWJ_LINEAR, dR, dS, dT, mode=m))
    hs = torch.cuda.current_stream().cuda_stream
    rel = binding._rel
    ctx._check(ctx.lib.mwj_join3_linear(ctx.h, rel(dR), rel(dS), rel(dT), None, ctypes.byref(o), ws.data_ptr(),
                                        ws.numel(), hs))
    with pytest.raises(binding.MwjError) as e:
        ctx._check(ctx.lib.mwj_stream_status(ctx.h, hs))
    assert e.value.status == binding.MWJ_ERR_CAPACITY and int(res["n_rows"].item()) == n
    assert int((res["rows"][n - short:] != -7).sum().item()) == 0
