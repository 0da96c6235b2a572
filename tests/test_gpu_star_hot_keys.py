"""Star aggregates on few keys in R: tables at the edges of their spread-out
layouts, in both layouts and mixed, with keys that repeat, miss or are -1, against
the factorised sum; and hot keys cost no more than a million cold ones."""
import numpy as np
import pytest

from factorised import factorised_group_by
from paper_1905_13376_gb300 import binding

from gpu_util import cu

pytestmark = pytest.mark.gpu

DOM = 1 << 10
NS = (1 << 19) + 77   # facts: one more than the plan of small calls takes


@pytest.fixture(scope="module")
def ctx():
    import torch
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


def keys(kind, n):
    k = np.arange(-1, n - 1, dtype=np.int64)
    return (k if kind == "compact" else k * 7919 % (1 << 31) - 1).astype(np.int32)


# 2^14, 2^15, 2^17 keys and one more: a line, half a line, a pair of words per entry
@pytest.mark.parametrize("n", [1, 3, 1000, 4096, 16384, 16385, 32769, 131072, 131073])
@pytest.mark.parametrize("layout", ["compact", "wide", "mixed"])
def test_star_aggregates(ctx, n, layout):
    g = np.random.default_rng(n)
    b = keys("wide" if layout == "wide" else "compact", n)
    c = keys("compact" if layout == "compact" else "wide", n)
    R = (g.integers(0, DOM, n + n // 3).astype(np.int32), b[np.r_[np.arange(n), g.integers(0, n, n // 3)]])
    T = (c[g.integers(0, n, 2 * n)], g.integers(0, 50, 2 * n).astype(np.int32))
    hot = np.minimum(g.integers(0, n, NS), g.integers(0, n, NS))
    S = (b[hot], c[g.integers(0, n, NS)])
    miss = g.random(NS) < 0.2
    S[0][miss] = g.integers(-(1 << 31), 1 << 31, int(miss.sum())).astype(np.int32)
    total, cnt = factorised_group_by(R, S, T, DOM)
    d = [cu(x) for x in (R, S, T)]
    got = ctx.join3_star(*d, "group_by_a", a_domain=DOM)
    assert int(got["total"].item()) == total
    assert np.array_equal(got["counts"].cpu().numpy(), cnt)
    assert int(ctx.join3_star(*d, "count")["total"].item()) == total


def test_star_of_empty_relations(ctx):
    g = np.random.default_rng(0)
    S = tuple(g.integers(0, 50, NS).astype(np.int32) for _ in range(2))
    D = (g.integers(0, DOM, 60).astype(np.int32), g.integers(0, 50, 60).astype(np.int32))
    none = (np.zeros(0, np.int32),) * 2
    for R, T in ((none, D), (D, none), (none, none)):
        for mode in ("count", "group_by_a"):
            assert int(ctx.join3_star(cu(R), cu(S), cu(T), mode, a_domain=DOM)["total"].item()) == 0


@pytest.mark.parametrize("mode", ["count", "group_by_a"])
@pytest.mark.parametrize("wide", [False, True])
def test_hot_keys_cost_no_more_than_cold_ones(ctx, mode, wide):
    """2^24 facts in no order, on 1000 keys and on 2^20."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    n = 1 << 24

    def time(nd):
        spread = (lambda x: x * 7919 % (1 << 31)) if wide else (lambda x: x)
        ri = lambda k, hi: torch.randint(0, hi, (k,), generator=g, device="cuda", dtype=torch.int64)
        key = spread(torch.arange(nd, device="cuda")).to(torch.int32)
        R, T = (ri(nd, DOM).to(torch.int32), key), (key.clone(), ri(nd, 100).to(torch.int32))
        S = (spread(ri(n, nd)).to(torch.int32), spread(ri(n, nd)).to(torch.int32))
        ts = []
        for k in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            ctx.join3_star(R, S, T, mode, a_domain=DOM, sync=False)
            e1.record()
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        return sorted(ts[2:])[2]

    assert time(1000) < 1.3 * time(1 << 20)
