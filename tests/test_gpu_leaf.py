"""The float64 leaf of the Cholesky inverses at the edges of its 8-wide panels and 64-wide blocks."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sliced", [False, True])
@pytest.mark.parametrize("m", [1, 2, 7, 8, 9, 16, 31, 33, 63, 64, 65, 72, 127, 128, 129, 200])
def test_small_inverse(m, sliced):
    from paper_1312_1549_gb300.solver import spd_inverse
    rng = np.random.default_rng(m)
    Q, _ = np.linalg.qr(rng.standard_normal((m, m)))
    w = np.linspace(0.2, 4.0, m) if m > 1 else np.array([1.7])
    A = (Q * w) @ Q.T
    A = 0.5 * (A + A.T)
    P = spd_inverse(torch.from_numpy(A).to("cuda"), sliced=sliced).cpu().numpy()
    # Cholesky inverse: a few m kappa u |A^-1| (kappa 20); the sliced products add 2^-44 of theirs
    eps = 2.0 ** -53 if not sliced else 2.0 ** -44
    assert np.abs(P - np.linalg.inv(A)).max() <= 8 * m * 20 * 2.0 ** -53 * 5.0 + (8 * m * eps * 5.0 if sliced else 0.0)
    assert np.array_equal(P, P.T)


def test_pivot_is_reported():
    from paper_1312_1549_gb300._native import OMMError
    from paper_1312_1549_gb300.solver import spd_inverse
    A = np.eye(100)
    A[70, 70] = -1.0
    with pytest.raises(OMMError):
        spd_inverse(torch.from_numpy(A).to("cuda"))
