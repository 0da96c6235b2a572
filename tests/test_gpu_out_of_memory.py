"""Calls without shares whose default plan's workspace the device has no room for:
rows, chains of four and sketches then run the partitioned plan where that asks for
less, and raise where it does not."""
import numpy as np
import pytest
import torch

from paper_1905_13376_gb300 import binding

from gpu_util import cu, sorted_rows

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


def relations(k):
    g = np.random.default_rng(k)
    return [cu(tuple(g.integers(0, 30_000, 60_000).astype(np.int32) for _ in range(2))) for _ in range(k)]


CALLS = {
    "rows": (3, lambda c, d: torch.from_numpy(sorted_rows(c.join3_linear(*d, "rows", capacity=500_000)["rows"].cpu().numpy()))),
    "chain": (4, lambda c, d: c.join4_linear(*d, "group_by_a", a_domain=30_000)["counts"]),
    "sketches": (3, lambda c, d: c.fm_linear(*d, 30_000)["sketches"]),
}


@pytest.mark.parametrize("call", list(CALLS))
def test_default_plan_without_room(ctx, call):
    k, run = CALLS[call]
    d = relations(k)
    want = run(ctx, d)
    full = ctx._ws.numel()
    asked = []

    def room(most):
        def workspace(nbytes):
            asked.append(nbytes)
            if nbytes > most:
                raise torch.cuda.OutOfMemoryError("no room")
            return torch.empty(max(nbytes, 256), dtype=torch.uint8, device="cuda")
        return workspace

    ctx.workspace = room(full - 1)
    assert torch.equal(run(ctx, d), want)
    assert asked[0] == full and asked[-1] < full
    ctx.workspace = room(1000)
    with pytest.raises(torch.cuda.OutOfMemoryError):
        run(ctx, d)


def test_calls_with_shares_do_not_change_them(ctx):
    R, S, T = relations(3)
    ctx.workspace = lambda nbytes: (_ for _ in ()).throw(torch.cuda.OutOfMemoryError("no room"))
    for f in (lambda: ctx.fm_linear(R, S, T, 30_000, shares=(64, 1, 1)), lambda: ctx.join3_linear(R, S, T, "count"),
              lambda: ctx.join3_linear(R, S, T, "rows", shares=(8, 1), capacity=10)):
        with pytest.raises(torch.cuda.OutOfMemoryError):
            f()
