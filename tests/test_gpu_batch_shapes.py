"""How a batch's shares and kernels follow its size: few cyclic queries are cut into
more tiles than each of many, and batches of many small relations, of as large ones
as that kernel takes and of one more tuple count alike; against the oracle."""
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


def rels(g, n, d):
    return [(g.integers(0, d, k).astype(np.int32), g.integers(0, d, k).astype(np.int32)) for k in n]


def test_few_queries_are_cut_finer(ctx):
    g = np.random.default_rng(1)
    dev = [cu(r) for r in rels(g, (10_000,) * 3, 101)]
    tiles = {}
    for n in (1, 8, 400):
        b = binding.Batch(ctx, [(binding.MWJ_CYCLIC, *dev)] * n)
        tiles[n] = int(np.prod(b.shares(n - 1)))
        b.close()
    assert tiles[1] == tiles[8] >= 32 and tiles[400] <= tiles[1] // 2


@pytest.mark.parametrize("nq", [1, 8])
def test_few_queries(ctx, nq):
    g = np.random.default_rng(nq)
    qs = [rels(g, (4000 + 100 * k, 5000, 4500), 71) for k in range(nq)]
    b = binding.Batch(ctx, [(binding.MWJ_CYCLIC, *[cu(r) for r in q]) for q in qs])
    got = b.launch().cpu().numpy()
    assert np.array_equal(got, [oracle.cyclic(*q)["total"] for q in qs])
    b.close()


def test_dense_keys_cost_little_more_than_sparse_ones(ctx):
    """One query of 1e4 tuples a relation: 1e6 wedges over the GPU, not over 8 tiles."""
    import torch

    def time(d):
        g = np.random.default_rng(d)
        b = binding.Batch(ctx, [(binding.MWJ_CYCLIC, *[cu(r) for r in rels(g, (10_000,) * 3, d)])])
        ts = []
        for k in range(9):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            b.launch()
            e1.record()
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        b.close()
        return sorted(ts[3:])[2]

    assert time(101) < 2.5 * time(10_000)


@pytest.mark.parametrize("most", [700, 16384, 16385])
def test_many_small_relations(ctx, most):
    g = np.random.default_rng(most)
    qs = []
    for k in range(400):
        n = [int(x) for x in 2 ** g.uniform(0, 9.5, 3)]
        if k == 7:
            n[most % 3] = most
        qs.append((binding.MWJ_CYCLIC if k % 4 == 1 else binding.MWJ_LINEAR, *rels(g, n, 40)))
    b = binding.Batch(ctx, [(q[0], *[cu(r) for r in q[1:]]) for q in qs])
    want = [(oracle.cyclic if q[0] == binding.MWJ_CYCLIC else oracle.linear)(*q[1:])["total"] for q in qs]
    for _ in range(2):
        assert np.array_equal(b.launch().cpu().numpy(), want)
    b.close()
