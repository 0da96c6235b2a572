"""Row output of the C-bucket plan when one warp step makes 2^32 rows and more: a
(c, a) pair that T holds 2^27 times and lists that hold its a 32 times and more.
The number of rows is exact, and nothing but rows[0, capacity) is written."""
import ctypes

import pytest

from paper_1905_13376_gb300 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("c,a", [(5, 7), (-1, -1)])
@pytest.mark.parametrize("copies,extra", [(32, 0), (128, 0), (33, 12345)])
def test_rows_of_a_step_past_32_bits(copies, extra, c, a):
    import torch
    torch.cuda.set_device(0)
    ctx = binding.Context(0)
    nt = (1 << 27) + extra
    col = lambda n, v: torch.full((n,), v, dtype=torch.int32, device="cuda")
    R, S, T = (col(copies, a), col(copies, 3)), (col(1, 3), col(1, c)), (col(nt, c), col(nt, a))
    want = copies * nt
    assert want >= 1 << 32
    mode, cap = binding.MODES["rows"], 100
    o, res = ctx._outputs(mode, None, cap + 100, 3)
    o.capacity = cap
    res["rows"].fill_(-9)
    sh = binding._shares((1, 1, 1))
    rel = [binding._rel(x) for x in (R, S, T)]
    ws = ctx.workspace(ctx.workspace_size(binding.MWJ_CYCLIC, R, S, T, shares=(1, 1, 1), mode=mode))
    hs = torch.cuda.current_stream().cuda_stream
    ctx._check(ctx.lib.mwj_join3_cyclic(ctx.h, *rel, sh, ctypes.byref(o), ws.data_ptr(), ws.numel(), hs))
    assert ctx.lib.mwj_stream_status(ctx.h, hs) == binding.MWJ_ERR_CAPACITY
    assert int(res["n_rows"].item()) == want and int(res["total"].item()) == want
    row = torch.tensor([a, 3, c], dtype=torch.int32, device="cuda")
    assert bool((res["rows"][:cap] == row).all()) and bool((res["rows"][cap:] == -9).all())
    assert int(ctx.join3_cyclic(R, S, T, "count", shares=(1, 1, 1))["total"].item()) == want
    ctx.close()
