"""The C-bucket probe's queue of long lists: items of as many S tuples as it has
places and one more (those share lists of 128 entries, larger items only lists of
2048), an item with more long lists than places, a second round over the queue.
Against sums over the (b, c) pairs; and the time of few tuples with long lists."""
import numpy as np
import pytest
import torch

from paper_1905_13376_gb300 import binding

from gpu_util import cu, sorted_rows

pytestmark = pytest.mark.gpu

NA = 4000


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


def lists(lens, seed):
    """R with a list of lens[b] different a values for every b."""
    g = np.random.default_rng(seed)
    b = np.repeat(np.arange(len(lens)), lens).astype(np.int32)
    a = np.concatenate([g.permutation(NA)[:n] for n in lens]).astype(np.int32)
    return a, b


@pytest.mark.parametrize("lens", [(2047, 2048, 2049), (2100, 3000, 40), (127, 128, 129), (255, 256, 257, 383)])
@pytest.mark.parametrize("per_item", [40, 384, 385, 640, 768, 769, 1000])
def test_queue(ctx, lens, per_item):
    items = 4 * 2 * torch.cuda.get_device_properties(0).multi_processor_count
    n = per_item * items - 5
    g = np.random.default_rng(per_item)
    R = lists(lens, per_item)
    nb, nc = len(lens) + 1, 3
    S = (g.integers(0, nb, n).astype(np.int32), g.integers(0, nc, n).astype(np.int32))
    # about two closed wedges per tuple; each pair of T once
    p = g.permutation(nc * NA)[:nc * NA // 1000]
    T = ((p // NA).astype(np.int32), (p % NA).astype(np.int32))
    inR = np.zeros((nb, NA), np.int64)
    np.add.at(inR, (R[1], R[0]), 1)
    inT = np.zeros((nc, NA), np.int64)
    np.add.at(inT, (T[0], T[1]), 1)
    nS = np.zeros((nb, nc), np.int64)
    np.add.at(nS, (S[0], S[1]), 1)
    want = np.einsum("ba,ca,bc->a", inR, inT, nS)
    total = int(want.sum())
    d = [cu(x) for x in (R, S, T)]
    got = ctx.join3_cyclic(*d, "group_by_a", shares=(1, 1, 1), a_domain=NA)
    assert int(got["total"].item()) == total
    assert np.array_equal(got["counts"].cpu().numpy(), want)
    if per_item in (384, 385, 1000):
        rows = ctx.join3_cyclic(*d, "rows", shares=(1, 1, 1), capacity=total)
        assert int(rows["n_rows"].item()) == total
        rows = rows["rows"].cpu().numpy().astype(np.int64)
        key, cnt = np.unique((rows[:, 0] * nb + rows[:, 1]) * nc + rows[:, 2], return_counts=True)
        a, b, c = key // (nb * nc), key // nc % nb, key % nc
        assert np.array_equal(cnt, nS[b, c]) and (inR[b, a] * inT[c, a] == 1).all()
        assert len(key) == int(((inR[:, None, :] * inT[None, :, :]) * (nS > 0)[:, :, None]).sum())


def test_few_tuples_with_long_lists(ctx):
    """Zipf keys: an item of 32 S tuples holds lists of a thousand entries, which
    one warp walked alone."""
    n, al = 3000, 1.5

    def zipf(dom, seed):
        w = np.cumsum(np.arange(1, dom + 1, dtype=np.float64) ** -al)
        return np.searchsorted(w / w[-1], np.random.default_rng(seed).random(n)).clip(0, dom - 1).astype(np.int32)

    dom = n // 8
    d = [cu((zipf(dom, 2 * k), zipf(dom, 2 * k + 1))) for k in range(3)]
    flat = [cu(tuple(np.random.default_rng(s).permutation(np.arange(n) % dom).astype(np.int32) for s in (k, k + 9)))
            for k in range(3)]

    def time(rel):
        ts = []
        for k in range(9):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            ctx.join3_cyclic(*rel, "count", sync=False)
            e1.record()
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        return sorted(ts[3:])[2]

    wedges = lambda rel: int((torch.bincount(rel[0][1], minlength=dom) * torch.bincount(rel[1][0], minlength=dom)).sum())
    # a call without wedges worth mentioning, and 5e9 wedges a second on top
    assert time(d) < time(flat) + wedges(d) / 5e9 * 1e3
