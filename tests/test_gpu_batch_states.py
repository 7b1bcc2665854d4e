"""The float64 recomputes of a batch's small instances run as one launch per step: uneven sizes (tiles of 16
and 32 with remainders) and real forms against the eigenpair definition."""
import numpy as np
import pytest
import torch

from oracle import exact

pytestmark = pytest.mark.gpu


def pencil(m, n, rng, complex_=False):
    z = (lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)) if complex_ else (lambda *s: rng.standard_normal(s))
    Q, _ = np.linalg.qr(z(m, m))
    w = np.concatenate([-2.0 + 0.5 * rng.random(n), 0.5 + rng.random(m - n)])
    R = np.eye(m) + 0.05 * z(m, m) / np.sqrt(m)
    S, H = R @ R.conj().T, R @ ((Q * w) @ Q.conj().T) @ R.conj().T
    return 0.5 * (H + H.conj().T), 0.5 * (S + S.conj().T), 2.0 * w[:n].sum(), 0.1 * z(n, m) / np.sqrt(m)


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def test_uneven_small_instances():
    from paper_1312_1549_gb300 import OMMBatch
    rng = np.random.default_rng(5)
    sizes = [(3, 1), (15, 4), (16, 16 // 2), (17, 5), (33, 31), (64, 32), (95, 17), (130, 33)]
    ps = [pencil(m, n, rng) for m, n in sizes]
    with OMMBatch([(dev(H), dev(S), dev(np.eye(m)), n, 0.0, 5.0) for (m, n), (H, S, _, _) in zip(sizes, ps)]) as b:
        _, E, _ = b.solve([dev(p[3]) for p in ps])
        D = [b.backward(i) for i in range(len(ps))]
    for i, ((m, n), (H, S, Eex, _)) in enumerate(zip(sizes, ps)):
        ex = exact.exact_minimum(H, S, n)
        assert abs(E[i] - Eex) <= 1e-9 * abs(Eex)
        assert np.abs(D[i][0].cpu().numpy() - ex["D"]).max() <= 1e-7
        assert np.abs(D[i][1].cpu().numpy() + ex["EDM"]).max() <= 1e-6


def test_hermitian_instances():
    from paper_1312_1549_gb300 import OMMHermitianBatch
    rng = np.random.default_rng(6)
    sizes = [(5, 2), (16, 7), (23, 11), (40, 9)]
    ps = [pencil(m, n, rng, True) for m, n in sizes]
    with OMMHermitianBatch([(dev(H), dev(S), dev(np.eye(m).astype(complex)), n, 0.0, 5.0)
                            for (m, n), (H, S, _, _) in zip(sizes, ps)]) as b:
        _, E, _ = b.solve([dev(p[3]) for p in ps])
        D = [b.backward(i) for i in range(len(ps))]
    import scipy.linalg
    for i, ((m, n), (H, S, Eex, _)) in enumerate(zip(sizes, ps)):
        w, X = scipy.linalg.eigh(H, S)
        X = X[:, :n]
        assert abs(E[i] - Eex) <= 1e-9 * abs(Eex)
        assert np.abs(D[i][0].cpu().numpy() - 2.0 * X @ X.conj().T).max() <= 1e-7
        assert np.abs(D[i][1].cpu().numpy() + 2.0 * (X * w[:n]) @ X.conj().T).max() <= 1e-6
