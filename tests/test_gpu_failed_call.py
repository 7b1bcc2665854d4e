"""A call that the host refuses leaves nothing behind for the next one."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_next_call_after_a_refused_launch():
    from paper_1312_1549_gb300._native import OMMError
    from paper_1312_1549_gb300.solver import dgemm
    one = torch.ones((1, 1), device="cuda", dtype=torch.float64)
    rows = 64 * 65535 + 1  # one tile row more than a grid has: the launch itself is refused
    tall = torch.ones((rows, 1), device="cuda", dtype=torch.float64)
    with pytest.raises(OMMError):
        dgemm(0, 0, tall, one, torch.empty_like(tall))
    out = torch.zeros_like(one)
    dgemm(0, 0, one, one, out)
    assert out.item() == 1.0
