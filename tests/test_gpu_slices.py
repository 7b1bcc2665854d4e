"""Fixed-point slicing over the row lengths where its thread layout changes, odd leading dimensions and
extreme row scales, through the float64-class product."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def product(A, B, slices=10):
    from paper_1312_1549_gb300.solver import gemm_emu
    dev = torch.device("cuda")
    C = torch.empty((A.shape[0], B.shape[0]), dtype=torch.float64, device=dev)
    gemm_emu(torch.from_numpy(A).to(dev), torch.from_numpy(B).to(dev), C, slices=slices)
    return C.cpu().numpy()


@pytest.mark.parametrize("K", [1, 3, 4, 127, 128, 129, 512, 515, 2047, 2050, 8192, 8199, 16384])
def test_row_lengths(K):
    rng = np.random.default_rng(K)
    A = rng.standard_normal((37, K)) * np.exp(-8 * rng.random((37, K)))
    B = rng.standard_normal((21, K)) * np.exp(-8 * rng.random((21, K)))
    A[3] = 0.0
    A[5] *= 2.0 ** -30
    B[4] *= 2.0 ** 80
    want = A.astype(np.longdouble) @ B.astype(np.longdouble).T
    # a slice residual is below 2^-49 of its row's maximum and the dropped slice pairs below 2^-44.8 of
    # both maxima, per product
    bound = K * 2.0 ** -44 * np.abs(A).max(1)[:, None] * np.abs(B).max(1)[None, :]
    assert (np.abs(product(A, B) - want) <= bound).all()


@pytest.mark.parametrize("slices", [1, 2, 9, 10])
def test_integers_are_exact(slices):
    # entries of at most 5 slices - 1 bits below a common power of two are represented exactly, so the
    # product of two such matrices with one operand of a single slice is exact
    rng = np.random.default_rng(slices)
    A = rng.integers(-(2 ** (5 * slices - 2)) + 1, 2 ** (5 * slices - 2), (40, 200)).astype(np.float64)
    A[:, 0] = 2.0 ** (5 * slices - 2) - 1
    B = np.eye(200)[:50]
    assert np.array_equal(product(A, B, slices), A[:, :50])


def test_row_scales_outside_float32():
    # unit slices outside the float32 range fall to the general conversion: still the right product
    A = np.array([[1.0, 0.5], [3.0, -0.75]]) * 2.0 ** 100
    B = np.array([[1.0, 2.0], [0.25, -1.0]]) * 2.0 ** -60
    assert np.array_equal(product(A, B), A @ B.T)
