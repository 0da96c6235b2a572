"""Keys of the last relation that hold much of it in no order: counted right in
chains of three and four, next to light keys, in runs, and where the column is the
weights' own; and in little more time than keys that hold little."""
import pytest
import torch

from paper_1905_13376_gb300 import binding

pytestmark = pytest.mark.gpu

N = (1 << 19) + 1111
KEYS = 50_000


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


def column(n, kind, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randint(0, KEYS, (n,), generator=g, device="cuda", dtype=torch.int64)
    p = torch.rand(n, generator=g, device="cuda")
    if kind == "few":        # two keys have nearly all
        x = torch.where(p < 0.98, x % 2 + 7, x)
    elif kind == "many":     # 130 keys, most of them just above what counts as heavy
        x = torch.where(p < 0.9, x % 130, x)
    elif kind == "runs":     # runs across lanes and blocks
        x = torch.where(p < 0.5, x % 3, x).view(-1)
        x = torch.where(torch.arange(n, device="cuda") // 37 % 3 == 0, torch.full_like(x, 5), x)
    elif kind == "one":
        x = torch.full_like(x, KEYS - 1)
    return (x - 100).to(torch.int32)


@pytest.mark.parametrize("kind", ["few", "many", "runs", "one"])
@pytest.mark.parametrize("same", [False, True])
def test_heavy_degrees(ctx, kind, same):
    c = column(N, kind, 1)
    b = c if same else column(N, "light", 2)
    a, y = column(N, "light", 3) % 1000, column(N, "light", 4)
    a = (a + 1000) % 1000
    R, S, T = (a, column(N, kind, 5)), (b, y), (c, y)
    rank = lambda x: x.long() + 100
    deg = torch.bincount(rank(c), minlength=KEYS)
    w = torch.bincount(rank(b), weights=deg[rank(y)].double(), minlength=KEYS)
    want = torch.bincount(a, weights=w[rank(R[1])], minlength=1000).to(torch.int64)
    assert torch.equal(ctx.join3_linear(R, S, T, "group_by_a", a_domain=1000)["counts"], want)
    w2 = torch.bincount(rank(b), weights=w[rank(y)], minlength=KEYS)
    want = torch.bincount(a, weights=w2[rank(R[1])], minlength=1000).to(torch.int64)
    assert float(w2.max().item()) < 2.0 ** 52
    assert torch.equal(ctx.join4_linear(R, S, S, T, "group_by_a", a_domain=1000)["counts"], want)


def test_two_keys_in_no_order_take_little_longer(ctx):
    n = 1 << 22
    light = [column(n, "light", k) for k in range(5)]

    def time(c):
        ts = []
        for k in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            ctx.join3_linear((light[0], light[1]), (light[2], light[3]), (c, light[4]), "count", sync=False)
            e1.record()
            torch.cuda.synchronize()
            ts.append(e0.elapsed_time(e1))
        return sorted(ts[2:])[2]

    assert time(column(n, "few", 9)) < 2 * time(column(n, "light", 9))
