"""Row output of relations too large for lists whose entries are numbered in 31
bits: they run the partitioned plan, and ask for its workspace."""
import ctypes

import pytest
import torch

from paper_1905_13376_gb300 import binding

pytestmark = pytest.mark.gpu

ROWS = binding.MODES["rows"]


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("large", [0, 2])
def test_workspace(ctx, large):
    def need(n, shares):
        sizes = [1000, 1000, 1000]
        sizes[large] = n
        rel = [binding.mwj_rel(0x10000 * (2 * k + 1), 0x10000 * (2 * k + 2), x) for k, x in enumerate(sizes)]
        sh, out = binding.mwj_shares(), ctypes.c_size_t()
        ctx._check(ctx.lib.mwj_plan_shares(ctx.h, binding.MWJ_LINEAR, *rel, ROWS, ctypes.byref(sh), None))
        ctx._check(ctx.lib.mwj_workspace_size(ctx.h, binding.MWJ_LINEAR, *rel, ctypes.byref(sh) if shares else None, ROWS,
                                              ctypes.byref(out)))
        return out.value

    assert need((1 << 29) - 1, False) != need((1 << 29) - 1, True)   # (another plan)
    for n in (1 << 29, (1 << 30) + 1, (1 << 31) - 1):
        assert need(n, False) == need(n, True)


def test_rows_of_a_billion_tuples(ctx):
    if torch.cuda.mem_get_info()[0] < 120 << 30:
        pytest.skip("needs 120 GB of device memory")
    n = (1 << 30) + 1
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    b = torch.empty(n, dtype=torch.int32, device="cuda")
    for i in range(0, n, 1 << 26):   # keys over the whole range, some twice
        m = min(1 << 26, n - i)
        b[i:i + m] = torch.randint(-(1 << 31), 1 << 31, (m,), generator=g, device="cuda", dtype=torch.int64).to(torch.int32)
    b[0], b[1] = -(1 << 31), (1 << 31) - 1
    R = (torch.arange(n, device="cuda", dtype=torch.int32), b)
    at = torch.randint(0, n, (500,), generator=g, device="cuda")
    S = (torch.cat([b[at], b[:2]]), torch.full((502,), 3, dtype=torch.int32, device="cuda"))
    T = (torch.full((2,), 3, dtype=torch.int32, device="cuda"), torch.tensor([8, 9], dtype=torch.int32, device="cuda"))
    # R's tuples with a key of S, and how often S holds each
    key, cnt = torch.unique(S[0], return_counts=True)
    hits = torch.cat([torch.nonzero(torch.isin(b[i:i + (1 << 27)], key)).flatten() + i for i in range(0, n, 1 << 27)])
    want = 2 * int(cnt[torch.searchsorted(key, b[hits])].sum().item())
    got = ctx.join3_linear(R, S, T, "rows", capacity=want + 10)
    assert int(got["n_rows"].item()) == want
    rows = got["rows"]
    assert bool((b[rows[:, 0].to(torch.int64)] == rows[:, 1]).all()) and bool((rows[:, 2] == 3).all())
    assert torch.equal(torch.unique(rows[:, 0]), torch.sort(hits.to(torch.int32))[0])
    assert int((rows[:, 3] == 8).sum().item()) == want // 2
    ctx._ws = None
