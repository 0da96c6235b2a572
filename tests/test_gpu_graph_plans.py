"""Every plan that a call without shares takes, captured into a CUDA graph and
replayed on other data in the same buffers: the cluster launch of the smallest
chains, the four and the nine launches, stars, chains of four, sketches, row output
and cyclic joins of one edge list and of three relations."""
import numpy as np
import pytest
import torch

from paper_1905_13376_gb300 import binding

from gpu_util import cu, sorted_rows

pytestmark = pytest.mark.gpu

DOM = 5000


def data(n, k, seed, wide=False):
    g = np.random.default_rng(seed)
    out = [cu(tuple(g.integers(0, min(DOM, n), n).astype(np.int32) for _ in range(2))) for _ in range(k)]
    return [tuple(c * 7919 % (1 << 30) + 1 for c in r) for r in out] if wide else out


def agg(join, mode, k=3):
    dom = lambda r: {"a_domain": DOM} if mode == "group_by_a" else {}
    return lambda c, d, **kw: getattr(c, join)(*d[:k], mode, **dom(d), **kw)


CASES = {
    "cluster": (1000, False, agg("join3_linear", "group_by_a")),
    "four launches": (100_000, False, agg("join3_linear", "group_by_a")),
    "nine launches": (600_000, False, agg("join3_linear", "group_by_a")),
    "nine launches, hashed": (600_000, True, agg("join3_linear", "count")),
    "chain": (600_000, False, agg("join4_linear", "group_by_a", 4)),
    "small chain": (3000, False, agg("join4_linear", "count", 4)),
    "star count": (600_000, False, agg("join3_star", "count")),
    "star": (600_000, False, agg("join3_star", "group_by_a")),
    "star, hashed": (600_000, True, agg("join3_star", "count")),
    "rows": (20_000, False, lambda c, d, **kw: c.join3_linear(*d[:3], "rows", capacity=600_000, **kw)),
    "star rows": (20_000, False, lambda c, d, **kw: c.join3_star(*d[:3], "rows", capacity=600_000, **kw)),
    "sketches": (100_000, False, lambda c, d, **kw: c.fm_linear(*d[:3], DOM, **kw)),
    "sketches, hashed": (100_000, True, lambda c, d, **kw: c.fm_linear((d[0][0] % DOM, d[0][1]), *d[1:3], DOM, **kw)),
    "cyclic": (60_000, False, agg("join3_cyclic", "group_by_a")),
    "cyclic rows": (60_000, False, lambda c, d, **kw: c.join3_cyclic(*d[:3], "rows", capacity=600_000, **kw)),
    "one edge list": (60_000, False, lambda c, d, **kw: c.join3_cyclic(d[0], d[0], d[0][::-1], "count", **kw)),
    "one edge list, rows": (60_000, False,
                            lambda c, d, **kw: c.join3_cyclic(d[0], d[0], d[0][::-1], "rows", capacity=600_000, **kw)),
}


def result(out):
    if "sketches" in out:
        return [out["sketches"].cpu(), out["estimates"].cpu()]
    if "n_rows" in out:
        n = int(out["n_rows"].item())
        return [torch.from_numpy(sorted_rows(out["rows"][:n].cpu().numpy()))]
    return [out[k].cpu().clone() for k in ("total", "counts") if k in out]


@pytest.mark.parametrize("name", list(CASES))
def test_captured_and_replayed(name):
    torch.cuda.set_device(0)
    ctx = binding.Context(0)
    n, wide, call = CASES[name]
    sets = [data(n, 4, seed, wide) for seed in (1, 2, 3)]
    want = [result(call(ctx, d)) for d in sets]
    assert not all(torch.equal(a, b) for a, b in zip(want[0], want[1]))
    buf = [tuple(c.clone() for c in r) for r in sets[0]]
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        call(ctx, buf, stream=s)   # (sizes the workspace outside the capture)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        out = call(ctx, buf, stream=s, sync=False)
    for k in (1, 2, 0, 0):
        for r, q in zip(buf, sets[k]):
            for c, x in zip(r, q):
                c.copy_(x)
        g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(result(out), want[k]))
    assert ctx.lib.mwj_stream_status(ctx.h, None) == binding.MWJ_OK
    ctx.close()
