"""Partitioning into more than 4096 buckets (csrc/partition.cu, k_part_scatter_direct):
the CTAs' shared cursors at ragged sizes, with one bucket holding half of a
relation, and with the third column that row output of a self-join carries."""
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


def relations(n, seed, dom):
    g = np.random.default_rng(seed)
    dom = max(dom, 8)
    hot = lambda: np.where(g.random(n) < 0.5, 3, g.integers(0, dom, n)).astype(np.int32)
    some = lambda: g.integers(0, dom, n).astype(np.int32)
    a = g.integers(0, max(dom // 64, 2), n).astype(np.int32)
    return (a, some()), (some(), hot()), (hot(), a[::-1].copy())


# edges of a tile (4096 tuples), a CTA's several tiles, the first bucket count of this
# path, and the counts up to which one CTA scans them (4096 and 4 x 4096)
@pytest.mark.parametrize("z,n", [(4097, 1), (4097, 4095), (5000, 4097), (4097, 12289), (20011, 300001),
                                 (4096, 4000), (16383, 900), (16384, 900), (16385, 900)])
@pytest.mark.parametrize("self_join", [False, True])
def test_many_buckets(ctx, z, n, self_join):
    R, S, T = relations(n, z + n, n // 8 if self_join else n)
    if self_join:
        T = (R[1], R[0])
    dR, dS, dT = cu(R), cu(S), cu(T)
    if self_join:
        dT = (dR[1], dR[0])
    want = oracle.cyclic(R, S, T, oracle.COUNT)["total"]
    got = ctx.join3_cyclic(dR, dS, dT, "count", shares=(1, 1, z))
    assert int(got["total"].item()) == want
    rows = oracle.cyclic(R, S, T, oracle.MATERIALIZE, capacity=max(want, 1))["rows"]
    got = ctx.join3_cyclic(dR, dS, dT, "rows", shares=(1, 1, z), capacity=max(want, 1))
    assert int(got["n_rows"].item()) == want
    assert np.array_equal(sorted_rows(got["rows"].cpu().numpy()[:want]), rows)
