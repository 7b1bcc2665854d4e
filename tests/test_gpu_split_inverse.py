"""The split-form inverse at sizes that are not multiples of its 64-row blocks."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [129, 130, 191, 193, 255, 300, 449])
def test_contraction_ends_with_the_matrix(m):
    """A = d 1: Y = L^-1 = y 1 with y halfway between two bf16 numbers, so that every diagonal block of P = Y^T Y
    is a float32 leaf's y^2, to 2^-20. One stray row of the lo halves in the sums would add their square, 2^-16."""
    from paper_1312_1549_gb300.solver import spd_inverse
    y = 1.0 + 0.99 * 2.0 ** -8
    A = torch.eye(m, device="cuda", dtype=torch.float64) / y ** 2
    P = spd_inverse(A, slices=1).cpu().numpy()
    assert np.abs(np.diag(P) / y ** 2 - 1.0).max() <= 2.0 ** -20
    assert np.abs(P - np.diag(np.diag(P))).max() == 0.0
