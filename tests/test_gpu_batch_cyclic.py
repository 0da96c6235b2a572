"""Cyclic batch queries where the join kernel's choices change: each relation
the smallest or the largest (the wedge side), repeated pairs on every side,
chunks of R, S and T, the (-1, -1) pair, one hub key; against the oracle."""
import numpy as np
import pytest

import oracle
from paper_1905_13376_gb300 import binding

from gpu_util import cu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import torch
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


def queries(g):
    out = []

    def rel(n, xd, yd):
        return g.integers(0, xd, n).astype(np.int32), g.integers(0, yd, n).astype(np.int32)

    # every order of small, middle and large relations
    for n in [(300, 2500, 9000), (2500, 9000, 300), (9000, 300, 2500), (9000, 2500, 300), (300, 9000, 2500)]:
        out.append((rel(n[0], 60, 50), rel(n[1], 50, 70), rel(n[2], 70, 60)))
    # tiny domains: nearly every pair repeats on all sides; one tile of several chunks
    out.append((rel(5000, 9, 7), rel(6000, 7, 8), rel(7000, 8, 9)))
    # sizes at the chunk capacities
    for n in (2047, 2048, 2049):
        out.append((rel(n, 2000, 3), rel(1025, 3, 40), rel(n, 40, 2000)))
    # a hub: one b holds half of R and S
    b1 = np.where(g.random(4000) < 0.5, 5, g.integers(0, 900, 4000)).astype(np.int32)
    b2 = np.where(g.random(4000) < 0.5, 5, g.integers(0, 900, 4000)).astype(np.int32)
    out.append(((g.integers(0, 300, 4000).astype(np.int32), b1), (b2, g.integers(0, 200, 4000).astype(np.int32)),
                rel(5000, 200, 300)))
    # key -1 everywhere
    m = lambda n: np.where(g.random(n) < 0.5, -1, 3).astype(np.int32)
    out.append(((m(200), m(200)), (m(300), m(300)), (m(400), m(400))))
    return out


def test_cyclic_queries(ctx):
    qs = queries(np.random.default_rng(1))
    want = [oracle.cyclic(*q, oracle.COUNT)["total"] for q in qs]
    for shares in (None, (1, 1, 1), (2, 3, 2)):
        b = binding.Batch(ctx, [(binding.MWJ_CYCLIC,) + tuple(cu(r) for r in q) + (shares,) for q in qs])
        got = b.launch().cpu().tolist()
        assert got == want, (shares, got, want)
        b.close()


def test_reported_shares_are_the_querys_own(ctx):
    """The library may take a query from another corner; shares are reported for
    its own A, B and C, and a batch given them back counts the same."""
    qs = queries(np.random.default_rng(2))
    dev = [tuple(cu(r) for r in q) for q in qs]
    a = binding.Batch(ctx, [(binding.MWJ_CYCLIC,) + d for d in dev])
    b = binding.Batch(ctx, [(binding.MWJ_CYCLIC,) + d + (a.shares(i),) for i, d in enumerate(dev)])
    assert [b.shares(i) for i in range(len(qs))] == [a.shares(i) for i in range(len(qs))]
    assert a.launch().cpu().tolist() == b.launch().cpu().tolist()
