"""The C-bucket plan's on-chip set and its filter at their edges: T chunks of
6144 tuples, buckets that move to the L2 above 16384, R lists around the warp
step of 1024 and the queue's 512, repeated pairs and the (-1, -1) pair behind
the filter.  All results against the oracle, bit for bit."""
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


def check(ctx, R, S, T, a_domain, shares):
    want = oracle.cyclic(R, S, T, oracle.GROUP_BY_A, a_domain=a_domain)
    got = ctx.join3_cyclic(cu(R), cu(S), cu(T), "group_by_a", shares=shares, a_domain=a_domain)
    assert int(got["total"].item()) == want["total"]
    assert np.array_equal(got["counts"].cpu().numpy(), want["counts"])
    n = want["total"]
    rows = oracle.cyclic(R, S, T, oracle.MATERIALIZE, capacity=n)["rows"]
    got = ctx.join3_cyclic(cu(R), cu(S), cu(T), "rows", shares=shares, capacity=n)
    assert int(got["n_rows"].item()) == n
    assert np.array_equal(sorted_rows(got["rows"].cpu().numpy()), rows)
    return n


@pytest.mark.parametrize("nt", [6143, 6144, 6145, 7167, 7168, 7169, 12289, 16384, 16385])
def test_chunk_edges(ctx, nt):
    """One bucket holding nt T tuples: one, two and three on-chip chunks, and the
    L2 set."""
    g = np.random.default_rng(nt)
    a_dom = 3000
    T = (g.integers(0, 40, nt).astype(np.int32), g.integers(0, a_dom, nt).astype(np.int32))
    R = (g.integers(0, a_dom, 5000).astype(np.int32), g.integers(0, 30, 5000).astype(np.int32))
    S = (g.integers(0, 33, 300).astype(np.int32), g.integers(0, 44, 300).astype(np.int32))
    assert check(ctx, R, S, T, a_dom, (1, 1, 1)) > 0


@pytest.mark.parametrize("length", [1, 31, 32, 127, 128, 129, 511, 512, 1023, 1024, 1025, 2047, 3000])
def test_list_lengths(ctx, length):
    """Every b has a list of `length` a values: short, walked and queued lists,
    full and partial steps; more lists than the queue holds."""
    g = np.random.default_rng(length)
    nb, a_dom = 20, 8192
    R = (g.integers(0, a_dom, nb * length).astype(np.int32), np.repeat(np.arange(nb), length).astype(np.int32))
    S = (g.integers(0, nb + 2, 900).astype(np.int32), g.integers(0, 50, 900).astype(np.int32))
    T = (g.integers(0, 50, 6000).astype(np.int32), g.integers(0, a_dom, 6000).astype(np.int32))
    check(ctx, R, S, T, a_dom, (1, 1, 3))


def test_marker_pair_and_repeats(ctx):
    """(-1, -1) pairs (the empty marker, counted apart) and repeated pairs pass
    the filter like any other pair."""
    R = (np.full(300, -1, np.int32), np.arange(300, dtype=np.int32) % 3)
    S = (np.arange(600, dtype=np.int32) % 4, np.where(np.arange(600) % 2 == 0, -1, 7).astype(np.int32))
    T = (np.where(np.arange(90) % 3 == 0, -1, 7).astype(np.int32), np.full(90, -1, np.int32))
    want = oracle.cyclic(R, S, T, oracle.COUNT)["total"]
    assert want > 0
    for shares in ((1, 1, 1), (1, 1, 5), None):
        assert int(ctx.join3_cyclic(cu(R), cu(S), cu(T), "count", shares=shares)["total"].item()) == want


@pytest.mark.parametrize("seed", range(4))
def test_self_join_takes_the_shorter_list(ctx, seed):
    """T holds R's pairs with the columns exchanged (the same device columns):
    S's tuples are turned to their shorter list.  R a bag with repeats, S another
    relation or the same one, keys inside and outside R, -1 among them."""
    import torch
    g = np.random.default_rng(seed)
    dom = (40, 300, 2000, 90)[seed]
    n = (3000, 9000, 9000, 20000)[seed]
    a = g.integers(0, dom, n).astype(np.int32)
    b = np.minimum(g.integers(0, dom, n), g.integers(0, dom, n)).astype(np.int32)
    if seed == 3:
        b[g.random(n) < 0.1] = -1
    S = (g.integers(-1, dom + 5, 2500).astype(np.int32), g.integers(-1, dom + 5, 2500).astype(np.int32))
    x, y = cu((a, b))
    for own, dev in ((S, cu(S)), ((b, a), (y, x))):
        if len(own[0]) > 10000:
            continue   # (the oracle's walk)
        want = oracle.cyclic((a, b), own, (b, a), oracle.GROUP_BY_A, a_domain=dom)
        for shares in (None, (1, 1, 7), (2, 2, 2)):
            got = ctx.join3_cyclic((x, y), dev, (y, x), "group_by_a", shares=shares, a_domain=dom)
            assert int(got["total"].item()) == want["total"]
            assert np.array_equal(got["counts"].cpu().numpy(), want["counts"])
        n_rows = want["total"]
        if n_rows < 3_000_000:
            rows = oracle.cyclic((a, b), own, (b, a), oracle.MATERIALIZE, capacity=n_rows)["rows"]
            got = ctx.join3_cyclic((x, y), dev, (y, x), "rows", capacity=n_rows)
            assert np.array_equal(sorted_rows(got["rows"].cpu().numpy()), rows)


@pytest.mark.parametrize("mode", ["count", "rows"])
def test_self_join_in_a_workspace_of_other_buffers(ctx, mode):
    """A workspace sized for equal relations in buffers of their own has no room
    for the turned tuples; the self-join takes it all the same."""
    import ctypes
    import torch
    g = np.random.default_rng(5)
    a, b = (g.integers(0, 3000, 40_000).astype(np.int32) for _ in range(2))
    x, y = cu((a, b))
    m = binding.MODES[mode]
    nb = ctx.workspace_size(binding.MWJ_CYCLIC, (x, y), (x, y), (y.clone(), x.clone()), mode=m)
    assert nb < ctx.workspace_size(binding.MWJ_CYCLIC, (x, y), (x, y), (y, x), mode=m)
    want = oracle.cyclic((a, b), (a, b), (b, a), oracle.MATERIALIZE, capacity=200_000)
    o, res = ctx._outputs(m, None, 200_000, 3)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    hs = torch.cuda.current_stream().cuda_stream
    rel = binding._rel
    ctx._check(ctx.lib.mwj_join3_cyclic(ctx.h, rel((x, y)), rel((x, y)), rel((y, x)), None, ctypes.byref(o),
                                        ws.data_ptr(), nb, hs))
    ctx._check(ctx.lib.mwj_stream_status(ctx.h, hs))
    assert int(res["total"].item()) == want["total"]
    if mode == "rows":
        n = int(res["n_rows"].item())
        assert np.array_equal(sorted_rows(res["rows"][:n].cpu().numpy()), want["rows"][:n])


@pytest.mark.parametrize("copies", [1, 31, 33, 400])
def test_rows_staged_and_not(ctx, copies):
    """Row output at the staging's edges: pairs of T repeated below and above the
    32 rows that a warp stages, and a capacity that all but one row fits."""
    g = np.random.default_rng(copies)
    a, b, c = (g.integers(0, 200, 900).astype(np.int32) for _ in range(3))
    T = (np.repeat(c[:100], copies), np.repeat(a[:100], copies))
    R, S = (a, b), (b, c)
    want = oracle.cyclic(R, S, T, oracle.COUNT)["total"]
    rows = oracle.cyclic(R, S, T, oracle.MATERIALIZE, capacity=want)["rows"]
    got = ctx.join3_cyclic(cu(R), cu(S), cu(T), "rows", shares=(1, 1, 4), capacity=want)
    assert int(got["n_rows"].item()) == want and int(got["total"].item()) == want
    assert np.array_equal(sorted_rows(got["rows"].cpu().numpy()), rows)
    with pytest.raises(binding.MwjError) as ei:
        ctx.join3_cyclic(cu(R), cu(S), cu(T), "rows", shares=(1, 1, 4), capacity=want - 1)
    assert ei.value.status == binding.MWJ_ERR_CAPACITY and str(want) in str(ei.value)


def test_list_lengths_and_alignments(ctx):
    """Lists of every length around the warp's 32, the 128 and 256 entries of its
    loads and the 1024 of a step, one after the other, so that they start at all
    places of a 16-byte load; every a of a list's first and last entries closes."""
    g = np.random.default_rng(17)
    lens = np.r_[29:38, 124:134, 253:260, 508:516, 1020:1030, 2045:2051]
    b = np.repeat(np.arange(len(lens)), lens).astype(np.int32)
    a = np.concatenate([g.permutation(5000)[:n] for n in lens]).astype(np.int32)
    first = np.cumsum(lens) - lens
    ends = np.r_[first, first + 1, first + 2, first + 3, first + lens - 1, first + lens - 2, first + lens - 4]
    c = g.integers(0, 6, 300).astype(np.int32)
    S = (g.integers(0, len(lens) + 2, 300).astype(np.int32), c)
    T = (g.integers(0, 6, 2400).astype(np.int32), np.r_[a[ends], g.integers(0, 5000, 2400 - len(ends))].astype(np.int32))
    assert check(ctx, (a, b), S, T, 5000, (1, 1, 3)) > 0
    T = (np.repeat(np.arange(6, dtype=np.int32), len(ends)), np.tile(a[ends], 6))
    assert check(ctx, (a, b), S, T, 5000, (1, 1, 3)) >= 7 * 290
