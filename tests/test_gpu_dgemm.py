"""The float64 product over the sizes where its tile and contraction split change (1 to 8 CTAs of a
cluster, 16-, 32- and 64-wide tiles), all transpositions, strided outputs and beta, against numpy."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (16, 16, 32), (17, 15, 33), (36, 207, 207), (36, 144, 207), (64, 416, 416), (33, 65, 1000),
          (128, 256, 256), (200, 200, 64), (300, 700, 31), (1024, 1024, 129)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("trans", [(0, 0), (0, 1), (1, 0), (1, 1)])
def test_dgemm_sizes(shape, trans):
    from paper_1312_1549_gb300.solver import dgemm
    M, N, K = shape
    rng = np.random.default_rng(M * 7 + N * 3 + K)
    A, B, C = (rng.standard_normal(s) for s in ((M, K), (K, N), (M, N)))
    dev = torch.device("cuda")
    tA = torch.from_numpy(np.ascontiguousarray(A.T if trans[0] else A)).to(dev)
    tB = torch.from_numpy(np.ascontiguousarray(B.T if trans[1] else B)).to(dev)
    for alpha, beta in ((1.0, 0.0), (-2.5, 0.75)):
        out = torch.from_numpy(C.copy() if beta else np.full((M, N), np.nan)).to(dev)
        dgemm(trans[0], trans[1], tA, tB, out, alpha, beta)
        again = torch.from_numpy(C.copy() if beta else np.full((M, N), np.nan)).to(dev)
        dgemm(trans[0], trans[1], tA, tB, again, alpha, beta)
        want = alpha * (A.astype(np.longdouble) @ B.astype(np.longdouble)) + beta * C
        # K products and sums of any order, alpha, beta and the final add, each within half an ulp
        bound = (K + 4) * 2.0 ** -53 * (abs(alpha) * (np.abs(A) @ np.abs(B)) + abs(beta) * np.abs(C)) * 1.001
        assert (np.abs(out.cpu().numpy() - want) <= bound).all()
        assert torch.equal(out, again)  # fixed summation order
