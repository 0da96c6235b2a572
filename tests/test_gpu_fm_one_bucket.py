"""Flajolet-Martin sketches in one bucket: direct-address and hashed rows in
every pairing, key -1, ragged sizes, sorted and random order, unaligned
columns, and the partitioned plan on the same inputs.  Bit for bit."""
import numpy as np
import pytest
import torch

from oracle import fm
from paper_1905_13376_gb300 import binding

from gpu_util import cu

pytestmark = pytest.mark.gpu

SPREAD = lambda k: ((k * 2654435761 + 12345) % (1 << 32) - (1 << 31)).astype(np.int32)
DENSE = lambda k: (k - 1).astype(np.int32)   # key -1 among them
MARK = lambda k: np.where(k % 2 == 0, -1, (1 << 31) - 1 - k).astype(np.int32)


@pytest.fixture(scope="module")
def ctx():
    torch.cuda.set_device(0)
    c = binding.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("fb", [SPREAD, DENSE, MARK])
@pytest.mark.parametrize("fc", [SPREAD, DENSE, MARK])
@pytest.mark.parametrize("n", [1, 31, 33, 1000, 20011])
def test_layouts(ctx, fb, fc, n):
    g = np.random.default_rng(n)
    dom, adom = max(2, n // 6), 40
    b, c = np.sort(g.integers(0, dom, n)) if n % 2 else g.integers(0, dom, n), g.integers(0, dom, n)
    S = (fb(b), fc(c))
    R = (g.integers(0, adom, n + 5).astype(np.int32), fb(g.integers(0, dom, n + 5)))
    T = (fc(g.integers(0, dom, n + 1)), g.integers(-1000, 1000, n + 1).astype(np.int32))
    want, _ = fm.sketches(R, S, T, adom)
    off = []
    for r in (R, S, T):
        cols = []
        for col in r:
            t = torch.empty(len(col) + 1, dtype=torch.int32, device="cuda")
            t[1:] = torch.from_numpy(np.ascontiguousarray(col)).cuda()
            cols.append(t[1:])
        off.append(tuple(cols))
    for rels, shares in (((cu(R), cu(S), cu(T)), None), (off, None), ((cu(R), cu(S), cu(T)), (7,))):
        got = ctx.fm_linear(*rels, adom, shares=shares)
        assert np.array_equal(got["sketches"].cpu().numpy().view(np.uint32), want)
        assert np.allclose(got["estimates"].cpu().numpy(), [fm.estimate(w) for w in want], rtol=1e-6)


def test_domain_error_is_reported(ctx):
    R = (np.array([0, 9], np.int32), np.array([1, 1], np.int32))
    S = (np.array([1], np.int32), np.array([2], np.int32))
    T = (np.array([2], np.int32), np.array([3], np.int32))
    with pytest.raises(binding.MwjError) as e:
        ctx.fm_linear(cu(R), cu(S), cu(T), 5)
    assert e.value.status == binding.MWJ_ERR_DOMAIN
