"""A context that factors nothing (no preconditioner) reports no failed pivot, whatever its memory held before."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_no_preconditioner_after_a_failed_factorisation(precision):
    from paper_1312_1549_gb300 import _native as N, solver
    m, n = 48, 8
    rng = np.random.default_rng(3)
    q, _ = np.linalg.qr(rng.normal(size=(m, m)))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    H = dev(q @ np.diag(np.where(np.arange(m) < n, -1.0, 1.0)) @ q.T)
    S, T = dev(np.eye(m)), dev(np.eye(m))
    bad = dev(-2.0 * np.eye(m))  # S + T / tau is not positive definite: a pivot is recorded and the memory given back
    for _ in range(4):
        with pytest.raises(N.OMMError):
            solver.OMMSolver(H, bad, T, n, 0.0, 1.0, precision=precision)
        solver.OMMSolver(H, S, T, n, 0.0, 1.0, precision=precision, precondition=False).close()
