"""The GEMM epilogues where their 32 x 32 blocks meet an edge: ragged rows and columns, odd leading
dimensions, beta, against the exact bf16 product; and odd-sized mixed solves (stacked outputs whose
blocks meet inside a 32-wide run) against the eigenpair definition."""
import numpy as np
import pytest
import torch

from oracle import exact

pytestmark = pytest.mark.gpu


def bf16(x):
    return torch.from_numpy(x).to(torch.bfloat16).to(torch.float64).numpy()


@pytest.mark.parametrize("shape", [(1, 1, 64), (31, 33, 64), (32, 32, 70), (33, 31, 64), (128, 255, 64), (129, 257, 130),
                                   (160, 95, 200)])
@pytest.mark.parametrize("tile", [128, 256])
def test_edges(shape, tile):
    from paper_1312_1549_gb300.solver import gemm_tc, gemm_tc_pair
    M, N, K = shape
    rng = np.random.default_rng(M + N + K)
    A, B, C = (rng.standard_normal(s) for s in ((M, K), (N, K), (M, N)))
    dev = lambda a: torch.from_numpy(a.copy()).to("cuda")
    a, b = bf16(A), bf16(B)
    for alpha, beta in ((1.0, 0.0), (-1.5, 1.0), (2.0, 0.25)):
        want = alpha * (a @ b.T) + beta * C
        # K exact products summed in float32 (any order), and float64 roundings far below that
        bound = abs(alpha) * K * 2.0 ** -23 * (np.abs(a) @ np.abs(b).T) + 2.0 ** -50 * np.abs(want)
        for out in (gemm_tc(dev(A), dev(B), dev(C), alpha, beta, npass=1, tile_n=tile),
                    gemm_tc_pair(dev(A), dev(B), dev(C), alpha, beta, tile_n=tile, npass=1)):
            assert (np.abs(out.cpu().numpy() - want) <= bound).all()


@pytest.mark.parametrize("m,n", [(41, 7), (95, 33), (130, 32), (163, 17)])
def test_odd_mixed_solve(m, n):
    from paper_1312_1549_gb300 import OMMSolver
    rng = np.random.default_rng(m)
    # n well separated low states in a mildly non-orthogonal basis
    Q, _ = np.linalg.qr(rng.standard_normal((m, m)))
    w = np.concatenate([-2.0 + 0.5 * rng.random(n), 0.5 + rng.random(m - n)])
    R = np.eye(m) + 0.05 * rng.standard_normal((m, m)) / np.sqrt(m)
    S, H = R @ R.T, R @ ((Q * w) @ Q.T) @ R.T
    S, H, T = 0.5 * (S + S.T), 0.5 * (H + H.T), np.eye(m)
    C0 = 0.1 * rng.standard_normal((n, m)) / np.sqrt(m)
    ex = exact.exact_minimum(H, S, n)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda")
    with OMMSolver(dev(H), dev(S), dev(T), n, 0.0, 5.0, precision="mixed") as s:
        _, E, D, _ = s.solve(dev(C0), want_D=True)
    assert abs(E - ex["E"]) <= 1e-9 * abs(ex["E"])
    assert np.abs(D.cpu().numpy() - ex["D"]).max() <= 1e-7
