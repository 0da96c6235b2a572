"""Workspaces: what a call asks for grows with its sizes, and a call without
shares whose workspace was sized for the partitioned plan runs that plan."""
import ctypes

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


@pytest.mark.parametrize("kind", [binding.MWJ_LINEAR, binding.MWJ_CYCLIC, binding.MWJ_STAR])
@pytest.mark.parametrize("mode", [binding.MWJ_COUNT, binding.MWJ_COUNT_GROUP_BY_A])
def test_workspace_grows_with_the_sizes(ctx, kind, mode):
    edges = [0, 1, 1 << 14, (1 << 14) + 1, 1 << 19, (1 << 19) + 1, 1 << 20, 5 << 20]

    def need(*n):
        out = ctypes.c_size_t()
        rel = [binding.mwj_rel(0x10000 * (2 * k + 1), 0x10000 * (2 * k + 2), x) for k, x in enumerate(n)]
        ctx._check(ctx.lib.mwj_workspace_size(ctx.h, kind, *rel, None, mode, ctypes.byref(out)))
        return out.value

    for r in (100, 1 << 19, 1 << 20):
        for t in (100, 1 << 20):
            sizes = [need(r, s, t) for s in edges]
            assert sizes == sorted(sizes)
            sizes = [need(s, r, t) for s in edges]
            assert sizes == sorted(sizes)


def relations(n, k):
    g = np.random.default_rng(n)
    return [tuple(g.integers(0, n // 2, n).astype(np.int32) for _ in range(2)) for _ in range(k)]


def stream():
    import torch
    return torch.cuda.current_stream().cuda_stream


def test_rows_in_a_partitioned_workspace(ctx):
    import torch
    R, S, T = relations(60_000, 3)
    d = [cu(x) for x in (R, S, T)]
    m = binding.MODES["rows"]
    sh = ctx.plan_shares(binding.MWJ_LINEAR, *d, mode=m)
    nb = ctx.workspace_size(binding.MWJ_LINEAR, *d, shares=sh, mode=m)
    assert nb < ctx.workspace_size(binding.MWJ_LINEAR, *d, mode=m)
    n = oracle.linear(R, S, T)["total"]
    o, res = ctx._outputs(m, None, n, 4)
    ws = torch.empty(nb, dtype=torch.uint8, device="cuda")
    ctx._check(ctx.lib.mwj_join3_linear(ctx.h, *[binding._rel(x) for x in d], None, ctypes.byref(o), ws.data_ptr(), nb,
                                        stream()))
    ctx._check(ctx.lib.mwj_stream_status(ctx.h, stream()))
    assert int(res["n_rows"].item()) == n
    want = oracle.linear(R, S, T, oracle.MATERIALIZE, capacity=n)["rows"]
    assert np.array_equal(sorted_rows(res["rows"].cpu().numpy()), want)


def test_chain_in_a_partitioned_workspace(ctx):
    import torch
    rel = relations(60_000, 4)
    d = [cu(x) for x in rel]
    args = [binding._rel(x) for x in d]
    sh = ctx.plan_shares(binding.MWJ_LINEAR, *d[:3], mode=binding.MODES["rows"])
    nb, full = ctypes.c_size_t(), ctypes.c_size_t()
    ctx._check(ctx.lib.mwj_join4_workspace_size(ctx.h, *args, binding._shares(sh), 1, ctypes.byref(nb)))
    ctx._check(ctx.lib.mwj_join4_workspace_size(ctx.h, *args, None, 1, ctypes.byref(full)))
    assert nb.value < full.value
    want = ctx.join4_linear(*d, "group_by_a", a_domain=30_000)
    o, res = ctx._outputs(1, 30_000, 0, 4)
    ws = torch.empty(nb.value, dtype=torch.uint8, device="cuda")
    ctx._check(ctx.lib.mwj_join4_linear(ctx.h, *args, None, ctypes.byref(o), ws.data_ptr(), nb.value, stream()))
    ctx._check(ctx.lib.mwj_stream_status(ctx.h, stream()))
    assert int(res["total"].item()) == int(want["total"].item()) == oracle.linear4(*rel)["total"]
    assert torch.equal(res["counts"], want["counts"])


def test_sketches_in_a_partitioned_workspace(ctx):
    import torch
    rel = relations(60_000, 3)
    d = [cu(x) for x in rel]
    args = [binding._rel(x) for x in d]
    nb, full = ctypes.c_size_t(), ctypes.c_size_t()
    ctx._check(ctx.lib.mwj_fm_workspace_size(ctx.h, *args, binding._shares((1024, 1, 1)), ctypes.byref(nb)))
    ctx._check(ctx.lib.mwj_fm_workspace_size(ctx.h, *args, None, ctypes.byref(full)))
    assert nb.value < full.value
    want = ctx.fm_linear(*d, a_domain=30_000)["sketches"]
    got = torch.empty_like(want)
    ws = torch.empty(nb.value, dtype=torch.uint8, device="cuda")
    ctx._check(ctx.lib.mwj_fm_linear(ctx.h, *args, None, 30_000, got.data_ptr(), None, ws.data_ptr(), nb.value, stream()))
    ctx._check(ctx.lib.mwj_stream_status(ctx.h, stream()))
    assert torch.equal(got, want)
