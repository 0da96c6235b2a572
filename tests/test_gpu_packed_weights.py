"""Weights of several million keys in hash tables: packed slots from 2^24 slots on,
with sums past 2^32, a key -1, keys that hold much of S, repeated and single keys, in
chains of three and four, against sums over the keys' ranks."""
import pytest
import torch

from paper_1905_13376_gb300 import binding

pytestmark = pytest.mark.gpu

N = 9_000_001
DOM = 1000


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


def ranks(n, hi, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randint(0, hi, (n,), generator=g, device="cuda", dtype=torch.int64)


def key(r):   # rank 0 is key -1; the others lie anywhere in 31 bits
    return torch.where(r == 0, -1, r * 214_013 % (1 << 31)).to(torch.int32)


# about 4.0 million keys (2^23 slots), 4.7 (2^24) and 6 of them in use
@pytest.mark.parametrize("keys", [4_500_000, 6_300_000, 11_000_000])
@pytest.mark.parametrize("kind", ["light", "heavy", "wide"])
def test_chains(ctx, keys, kind):
    b, c, t, rb = ranks(N, keys, 1), ranks(N, keys, 2), ranks(N, keys, 3), ranks(N, keys, 4)
    if kind == "heavy":      # key -1 and two more hold much of S
        b = torch.where(ranks(N, 10, 5) < 4, b % 3, b)
    if kind == "wide":       # one c has 1.5e6 of T and is met by a tenth of S: w(b) up to 2^42
        t[:1_500_000] = 77
        c[ranks(N, 10, 6) == 0] = 77
        b[c == 77] %= 40
    a = ranks(N, DOM, 7)
    deg = torch.bincount(t, minlength=keys)
    w = torch.bincount(b, weights=deg[c].double(), minlength=keys)
    assert (float(w.max().item()) > 2 ** 33) == (kind == "wide")
    want = torch.bincount(a, weights=w[rb], minlength=DOM).to(torch.int64)
    R, S, T = (a.to(torch.int32), key(rb)), (key(b), key(c)), (key(t), a.to(torch.int32))
    got = ctx.join3_linear(R, S, T, "group_by_a", a_domain=DOM)
    assert torch.equal(got["counts"], want) and int(got["total"].item()) == int(want.sum().item())
    assert int(ctx.join3_linear(R, S, T, "count")["total"].item()) == int(want.sum().item())
    if kind == "wide":
        return   # (beyond what doubles hold)
    w2 = torch.bincount(rb, weights=w[b], minlength=keys)
    total = int((torch.bincount(c, minlength=keys).double() * w2).sum().item())
    assert total < 2 ** 52
    # R(A,B) = (a, c), S = (rb, b) with keys turned round, T = (b, c), U = T
    assert int(ctx.join4_linear((R[0], key(c)), (key(rb), key(b)), S, T, "count")["total"].item()) == total
