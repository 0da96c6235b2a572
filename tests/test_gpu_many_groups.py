"""Outputs of many groups or sketches, zeroed by a memset of their own: right at the
sizes where it begins, and written over, in linear and star joins and sketches."""
import pytest
import torch

from paper_1905_13376_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


def rel(n, x, y, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return tuple(torch.randint(0, d, (n,), generator=g, device="cuda", dtype=torch.int64).to(torch.int32) for d in (x, y))


@pytest.mark.parametrize("groups", [1 << 24, (1 << 24) + 1, (1 << 25) + 7])
@pytest.mark.parametrize("n", [700, 1 << 16, 600_000])
def test_groups(ctx, groups, n):
    R, S, T = rel(n, groups, 500, 1), rel(n, 500, 500, 2), rel(n, 500, 9, 3)
    deg = torch.bincount(T[0], minlength=500)
    w = torch.bincount(S[0], weights=deg[S[1].long()].double(), minlength=500)
    want = torch.bincount(R[0], weights=w[R[1].long()], minlength=groups).to(torch.int64)
    out = None
    for _ in range(2):
        out = ctx.join3_linear(R, S, T, "group_by_a", a_domain=groups, out=out)
        assert torch.equal(out["counts"], want)
        out["counts"].fill_(-3)
    assert torch.equal(ctx.join3_star(R, S, T, "group_by_a", a_domain=groups)["counts"], want)


@pytest.mark.parametrize("groups", [1 << 22, (1 << 22) + 1])
def test_sketches(ctx, groups):
    R, S, T = rel(5000, groups, 500, 1), rel(5000, 500, 500, 2), rel(5000, 500, 900, 3)
    junk = torch.full((2 * groups, 16), -1, dtype=torch.int32, device="cuda")   # (what the allocator hands out again)
    del junk
    got = ctx.fm_linear(R, S, T, groups)["sketches"]
    assert torch.equal(got, ctx.fm_linear(R, S, T, groups, shares=(64, 1, 1))["sketches"])
