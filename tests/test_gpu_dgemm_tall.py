"""Float64 products with more rows than a grid has rows of 16- or 32-row tiles."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(16 * 65535, 1, 1), (16 * 65535 + 1, 1, 1), (1100000, 3, 5), (32 * 65535 + 1, 2, 40)])
@pytest.mark.parametrize("transA", [0, 1])
def test_tall_product(M, N, K, transA):
    from paper_1312_1549_gb300.solver import dgemm
    g = torch.Generator(device="cuda").manual_seed(M + K)
    A = torch.randint(-9, 10, (M, K), generator=g, device="cuda").double()
    B = torch.randint(-9, 10, (K, N), generator=g, device="cuda").double()
    C = torch.full((M, N), float("nan"), device="cuda", dtype=torch.float64)
    dgemm(transA, 0, A.T.contiguous() if transA else A, B, C)
    assert torch.equal(C, (A[:, :, None] * B[None]).sum(1))  # whole numbers: exact in any order
