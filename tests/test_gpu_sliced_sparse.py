"""Block-sparse sliced products whose left-over tiles are short (the last column blocks of a triangular B)."""
import os

import numpy as np
import pytest
import torch

from native_build import compile_program, run_program

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def product(tmp_path_factory):
    from paper_1312_1549_gb300 import build
    lib = build.build()
    return compile_program("sliced_product.cu", tmp_path_factory.mktemp("native"), *build.ARCH, lib, "-Xlinker",
                           "-rpath=" + os.path.dirname(lib))


# one left-over tile of 256 x 256, its last column block with one K block, on 76, 75 and 74 pairs of SMs
@pytest.mark.parametrize("M,N", [(1664, 2624), (896, 4672), (1152, 3648)])
def test_short_left_over_tile(product, M, N):
    run_program(product, M, N)


def test_cholesky_flavour_restores_every_column():
    """C S C^T of the returned coefficients is the identity at the minimum (Sec. 2.1)."""
    import paper_1312_1549_gb300 as omm
    m, n = 2624, 1664
    g = torch.Generator(device="cuda").manual_seed(4)
    X = torch.randn((m, m), generator=g, device="cuda", dtype=torch.float64) / m ** 0.5
    S = torch.eye(m, device="cuda", dtype=torch.float64) + 0.1 * (X + X.T)
    d = torch.linspace(-3.0, -2.0, m, device="cuda", dtype=torch.float64)
    d[n:] += 5.0
    H = torch.diag(d) + 0.05 * (X + X.T)
    C0 = torch.randn((n, m), generator=g, device="cuda", dtype=torch.float64) * (0.1 / m ** 0.5)
    # (a shift above the whole spectrum: from a random start the functional is unbounded with a lower one)
    sv = omm.OMMSolver(H.contiguous(), S.contiguous(), None, n, 4.5, 1.0, precision="mixed", cholesky=True,
                       tol_grad=1e-8)
    C = sv.solve(C0)[0]
    assert np.abs((C @ S @ C.T - torch.eye(n, device="cuda", dtype=torch.float64)).cpu().numpy()).max() < 1e-7
