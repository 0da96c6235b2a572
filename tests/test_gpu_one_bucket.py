"""The one-bucket plan's tables where their layouts change: direct-address
arrays with gaps and at the largest range they are given to, hashed pairs and
groups of four, key -1, runs and random order, ragged sizes and unaligned
columns, chains of three and of four.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_1905_13376_gb300 import binding

from factorised import factorised_group_by
from gpu_util import cu

pytestmark = pytest.mark.gpu

LAYOUTS = {
    "compact": lambda k: k,
    "gaps": lambda k: 7 * k - 1000,                                  # a direct-address range, mostly unused
    "hashed": lambda k: (k * 2654435761 + 12345) % (1 << 32) - (1 << 31),
    "extremes": lambda k: np.where(k % 3 == 0, -1, np.where(k % 3 == 1, -(1 << 31) + k, (1 << 31) - 1 - k)),
}


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


def rel(g, n, xdom, ydom, fx, fy, sort=False):
    x, y = g.integers(0, xdom, n), g.integers(0, ydom, n)
    if sort:
        x = np.sort(x)
    return fx(x).astype(np.int32), fy(y).astype(np.int32)


def unaligned(r):
    """The same columns four bytes off a 16-byte boundary."""
    out = []
    for c in r:
        t = torch.empty(len(c) + 1, dtype=torch.int32, device="cuda")
        t[1:] = torch.from_numpy(np.ascontiguousarray(c)).cuda()
        out.append(t[1:])
    return tuple(out)


def same(got, want):
    assert int(got["total"].item()) == want["total"]
    if "counts" in got:
        assert np.array_equal(got["counts"].cpu().numpy(), want["counts"])


@pytest.mark.parametrize("layout", list(LAYOUTS))
@pytest.mark.parametrize("n", [1, 3, 127, 129, 4097, (1 << 14) - 1, (1 << 14) + 1, 70001, 600001])
def test_chains(ctx, layout, n):
    g = np.random.default_rng(n + 7 * len(layout))
    f = LAYOUTS[layout]
    ident = lambda k: k
    dom, adom = max(2, n // 5), 50
    R = rel(g, n, adom, dom, ident, f)
    S = rel(g, max(1, n - 1), dom, dom, f, f, sort=n % 2 == 0)
    T = rel(g, n + 2, dom, dom, f, f, sort=n % 4 == 1)
    U = rel(g, n, dom, 9, f, ident)
    # (the oracle walks every (R, S) pair and every (b, c, d): too many where one
    # key holds a third of a large relation)
    if layout == "extremes" and n > 100000:
        total, counts = factorised_group_by(R, S, T, adom)
        want = {"total": total, "counts": counts}
    else:
        want = oracle.linear(R, S, T, oracle.GROUP_BY_A, a_domain=adom)
    want4 = oracle.linear4(R, S, T, U, oracle.GROUP_BY_A, a_domain=adom) if layout != "extremes" or n < 5000 else None
    for take in (cu, unaligned):
        d = [take(x) for x in (R, S, T, U)]
        same(ctx.join3_linear(*d[:3], "group_by_a", a_domain=adom), want)
        same(ctx.join3_linear(*d[:3], "count"), want)
        if want4 is not None:
            same(ctx.join4_linear(*d, "group_by_a", a_domain=adom), want4)


@pytest.mark.parametrize("span", [(1 << 21) - 1, 1 << 21, (1 << 21) + 1])
def test_largest_direct_range(ctx, span):
    """2^20 tuples reserve 2^21 slots: a key range of exactly that many values is
    the largest direct-address one."""
    g = np.random.default_rng(span)
    n = 1 << 20
    k = g.integers(0, span, n)
    k[:2] = (0, span - 1)
    k = (k - 77).astype(np.int32)
    R = (g.integers(0, 64, n).astype(np.int32), g.permutation(k))
    S = (k, g.permutation(k))
    T = (g.permutation(k), np.zeros(n, np.int32))
    want = oracle.linear(R, S, T, oracle.GROUP_BY_A, a_domain=64)
    same(ctx.join3_linear(cu(R), cu(S), cu(T), "group_by_a", a_domain=64), want)


@pytest.mark.parametrize("layout", ["compact", "hashed", "extremes"])
@pytest.mark.parametrize("n", [12000, 100000, 700000])
def test_heavy_keys_and_wide_weights(ctx, layout, n):
    """A few keys hold most of S in no order (heavy sums) and weights pass 2^32,
    in chains of three and four, in each of the plans by size."""
    g = np.random.default_rng(5)
    f = LAYOUTS[layout]
    b = np.where(g.random(n) < 0.6, g.integers(0, 3, n), g.integers(0, 500, n))
    S = (f(b).astype(np.int32), f(np.zeros(n, np.int64)).astype(np.int32))
    nt = 10000 if n < 16384 else 200000
    T = (f(np.where(g.random(nt) < 0.9, 0, 5)).astype(np.int32), f(np.zeros(nt, np.int64)).astype(np.int32))
    R = (g.integers(0, 20, 900).astype(np.int32), f(g.integers(0, 500, 900)).astype(np.int32))
    want = oracle.linear(R, S, T, oracle.GROUP_BY_A, a_domain=20)
    assert nt < 200000 or want["total"] > 1 << 33
    same(ctx.join3_linear(cu(R), cu(S), cu(T), "group_by_a", a_domain=20), want)
    if n > 20000:
        return   # (the oracle walks every (b, c, d))
    U = (f(np.zeros(5000, np.int64)).astype(np.int32), np.zeros(5000, np.int32))
    want = oracle.linear4(R, S, T, U, oracle.GROUP_BY_A, a_domain=20)
    same(ctx.join4_linear(cu(R), cu(S), cu(T), cu(U), "group_by_a", a_domain=20), want)


@pytest.mark.parametrize("lr", list(LAYOUTS))
@pytest.mark.parametrize("lt", list(LAYOUTS))
@pytest.mark.parametrize("n", [1, 130, 30001, 600001])
def test_star_keeps_only_r_keys(ctx, lr, lt, n):
    """Star joins lay the weights out for R's keys: S tuples inside and outside
    R's range, heavy ones among them, in every layout of both dimensions."""
    g = np.random.default_rng(n)
    fr, ft = LAYOUTS[lr], LAYOUTS[lt]
    dim = max(1, n // 30)
    R = (g.integers(0, 25, dim).astype(np.int32), fr(np.arange(dim) * 2).astype(np.int32))
    T = (ft(g.integers(0, 2 * dim, 2 * dim)).astype(np.int32), g.integers(0, 9, 2 * dim).astype(np.int32))
    b = np.where(g.random(n) < 0.4, 4 * dim, g.integers(0, 5 * dim, n))
    S = (fr(np.sort(b) if n % 2 else b).astype(np.int32), ft(g.integers(0, 3 * dim, n)).astype(np.int32))
    want = oracle.linear(R, S, T, oracle.GROUP_BY_A, a_domain=25)
    for take in (cu, unaligned):
        d = [take(x) for x in (R, S, T)]
        same(ctx.join3_star(*d, "group_by_a", a_domain=25), want)
        same(ctx.join3_star(*d, "count"), want)
