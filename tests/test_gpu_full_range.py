"""A key column of 2^30 + 1 tuples that holds the smallest and the largest 32-bit
value: its range is one more than 32 bits count."""
import pytest
import torch

from paper_1905_13376_gb300 import binding

pytestmark = pytest.mark.gpu


def test_all_32_bit_values():
    """2^30 + 1 tuples reserve 2^32 entries, which a column that holds the smallest
    and the largest key would need all."""
    if torch.cuda.mem_get_info()[0] < 120 << 30:
        pytest.skip("needs 120 GB of device memory")
    torch.cuda.set_device(0)
    ctx = binding.Context(0)
    n = (1 << 30) + 1
    x = torch.full((n,), 5, dtype=torch.int32, device="cuda")
    x[7], x[n - 2], x[11] = -(1 << 31), (1 << 31) - 1, -1
    S = (x, torch.full((n,), 9, dtype=torch.int32, device="cuda"))
    i32 = lambda *v: torch.tensor(v, dtype=torch.int32, device="cuda")
    R = (i32(0, 1, 2, 1, 0), i32(5, -(1 << 31), (1 << 31) - 1, -1, 6))
    T = (i32(9, 9, 8), i32(1, 2, 3))
    got = ctx.join3_linear(R, S, T, "group_by_a", a_domain=3)
    assert got["counts"].tolist() == [2 * (n - 3), 4, 2] and int(got["total"].item()) == 2 * n
    ctx.close()
