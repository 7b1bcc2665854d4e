"""The calls that users of the orbital minimization library make, as timed cases.

Each case is one pass through the Python entry points of `paper_1312_1549_gb300`:

  solve      OMMSolver: create, minimise, density matrix and dE/dS. The unit of work of a
             single-point calculation, in mixed precision or in float64, with the kinetic
             preconditioner or in the Cholesky flavour.
  scf        OMMSolver kept over the steps of a self-consistency loop: update_H, a solve started
             from the previous step's coefficients, and both gradients.
  autograd   omm_energy forward and backward (float64): E(H, S) inside a torch program.
  batch      OMMBatch: independent systems of uneven size (snapshots, spins), with their gradients.
  kpoints    OMMHermitianBatch: the points of a Brillouin-zone grid, with their density matrices.
  hermitian  OMMHermitian: one k point in float64.
  inverse    spd_inverse of S + T/tau: native float64, or float64-class on the tensor cores.
  gemm       gemm_emu: the float64-class product C = A B^T.
  dgemm      the float64 product in the layouts of the method's steps.

The matrices are those of finite-range atom-centred Gaussians: groups of s-type Gaussians at and
around the atoms (analytic overlaps S and kinetic integrals T, cut off smoothly at 9 bohr so that
distant blocks are exact zeros) and H = T - w B B^T + on-site noise, where the columns of B are the
overlaps with one attractive projector per occupied state. T is positive definite and B has n
columns, so the pencil (H, S) has n states below zero and a gap above them; the eigenspectrum shift
eta = 0 lies in it. Atoms sit on a diamond lattice (two occupied states per atom) or are molecules
on a disturbed cubic grid (four per molecule, 23 functions each, hence odd sizes), as in the
repository's silicon and water workloads, whose sizes the listed cases take.

The converged coefficients C are determined only up to a rotation among the occupied states, which
depends on the path of the minimisation; what a program goes on with is E, the density matrix D =
dE/dH and the energy-density matrix (dE/dS = -EDM), so those are the outputs. tol_grad is 1e-11
(forces and vibrations need that), which leaves D its float64 accuracy.
"""
import math

import numpy as np
import torch

import paper_1312_1549_gb300 as omm
from paper_1312_1549_gb300 import solver as steps

RC = 9.0            # range of the matrix elements, bohr
DEPTH = {"atoms": 1.9, "molecules": 3.2}   # strength of the projectors, hartree
NOISE = 0.01        # on-site noise, hartree
TAU = 5.0           # kinetic scale of the preconditioner, 10 Ry
ETA = 0.0
TOL = 1e-11
A_SI = 10.26        # silicon lattice constant, bohr

TETRA = np.array([[1, 1, 1], [1, -1, -1], [-1, 1, -1], [-1, -1, 1]]) / math.sqrt(3.0)
OCTA = np.array([[1, 0, 0], [0, 1, 0], [0, 0, 1], [-1, 0, 0], [0, -1, 0], [0, 0, -1]], float)
CENTRE = np.zeros((1, 3))

# groups of Gaussians of one atom or molecule: (exponent, distance from its centre, directions)
BASES = {
    4: [(0.33, 1.1, TETRA)],
    8: [(0.33, 1.1, TETRA), (0.9, 0.9, TETRA)],
    13: [(0.33, 1.1, TETRA), (0.9, 0.9, TETRA), (0.40, 2.2, OCTA[:5])],
    16: [(0.33, 1.1, TETRA), (0.9, 0.9, TETRA), (0.40, 2.2, OCTA[:5]), (2.4, 0.5, OCTA[:3])],
    23: [(0.7, 0.9, TETRA), (2.2, 0.8, TETRA), (0.5, 1.9, OCTA), (5.0, 0.35, TETRA), (0.30, 0.0, CENTRE),
         (1.2, 1.5, -TETRA)],
}
MOLECULE = 23       # this many functions: a molecule with four occupied states


def occupied(norb):
    return 4 if norb == MOLECULE else 2


def depth(norb):
    return DEPTH["molecules" if norb == MOLECULE else "atoms"]


def rotations(count, rng):
    q = rng.normal(size=(count, 4))
    q /= np.linalg.norm(q, axis=1)[:, None]
    w, x, y, z = q.T
    return np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                     2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                     2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], axis=1).reshape(count, 3, 3)


def geometry(units, norb, rng):
    """(centres, exponents) of the basis and of the projectors."""
    if norb == MOLECULE:
        k = math.ceil(units ** (1 / 3) - 1e-9)
        at = np.array([(i, j, l) for i in range(k) for j in range(k) for l in range(k)], float)[:units] * 5.87
        at += rng.uniform(-0.3, 0.3, size=at.shape)
        turn = rotations(units, rng)
        hold, wide = np.repeat((0.85 * TETRA)[None], units, 0), 0.75
    else:
        cells = math.ceil(units / 8)
        k = math.ceil(cells ** (1 / 3) - 1e-9)
        sub = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
        frac = np.concatenate([sub, sub + 0.25])
        cell = np.array([(i, j, l) for i in range(k) for j in range(k) for l in range(k)], float)[:cells]
        at = ((cell[:, None] + frac[None]).reshape(-1, 3) * A_SI)[:units]
        at += rng.normal(0.0, 0.05, size=at.shape)
        # the bonds of one sublattice point along TETRA, the other's along -TETRA; one projector per
        # bond: the first two bonds of the one's atoms, the last two of the other's
        first = (np.arange(units) % 8) < 4
        turn = np.where(first, 1.0, -1.0)[:, None, None] * np.eye(3)[None]
        half = TETRA * (A_SI * math.sqrt(3) / 8)
        hold, wide = np.where(first[:, None, None], half[None, :2], half[None, 2:]), 0.33
    offs = np.concatenate([r * d for _, r, d in BASES[norb]])
    expo = np.concatenate([np.full(len(d), a) for a, _, d in BASES[norb]])
    centres = (at[:, None] + np.einsum("uij,kj->uki", turn, offs)).reshape(-1, 3)
    proj = (at[:, None] + np.einsum("uij,ukj->uki", turn, hold)).reshape(-1, 3)
    return centres, np.tile(expo, units), proj, np.full(len(proj), wide)


def integrals(xa, ea, xb, eb, kinetic):
    """Overlaps (and kinetic integrals) of normalised s Gaussians, cut off at RC by a positive
    definite function, so that S and T stay positive definite."""
    d2 = sum((xa[..., :, None, k] - xb[..., None, :, k]) ** 2 for k in range(3))
    s, p = ea[:, None] + eb[None, :], ea[:, None] * eb[None, :]
    q = p / s
    u = torch.clamp(1.0 - torch.sqrt(d2) / RC, min=0.0)
    over = (2.0 * torch.sqrt(p) / s) ** 1.5 * torch.exp(-q * d2) * (u ** 4 * (5.0 - 4.0 * u))
    return (over, over * q * (3.0 - 2.0 * q * d2)) if kinetic else over


def generator(seed):
    return np.random.Generator(np.random.PCG64(np.random.SeedSequence([1312, int(seed)])))


def tensors(arrays, dev):
    return [torch.from_numpy(np.ascontiguousarray(a)).to(dev) for a in arrays]


def problem(units, norb, rng, dev):
    """(H, S, T, n, C0) of one system."""
    x, e, xp, ep = tensors(geometry(units, norb, rng), dev)
    m, n = len(e), len(ep)
    S, T = integrals(x, e, x, e, True)
    B = integrals(x, e, xp, ep, False)
    H = T - depth(norb) * (B @ B.T)
    H = 0.5 * (H + H.T)
    H.diagonal().add_(torch.from_numpy(rng.normal(0.0, NOISE, size=m)).to(dev))
    C0 = torch.from_numpy(rng.normal(0.0, 0.1, size=(n, m)) / math.sqrt(m)).to(dev)
    return H.contiguous(), S.contiguous(), T.contiguous(), n, C0


def bloch_problems(points, units, norb, rng, dev):
    """[(H, S, T, n, C0)] of `points` k points of a silicon cell of `units` atoms (eight: the cubic cell)."""
    x, e, xp, ep = tensors(geometry(units, norb, rng), dev)
    m, n = len(e), len(ep)
    edge = A_SI * math.ceil(math.ceil(units / 8) ** (1 / 3) - 1e-9)
    shifts = torch.tensor([(i, j, l) for i in (-1, 0, 1) for j in (-1, 0, 1) for l in (-1, 0, 1)],
                          dtype=torch.float64, device=dev) * edge
    S_R, T_R = integrals(x.expand(27, -1, -1), e, x[None] + shifts[:, None], e, True)
    B_R = integrals(x.expand(27, -1, -1), e, xp[None] + shifts[:, None], ep, False)
    noise = torch.from_numpy(rng.normal(0.0, NOISE, size=m)).to(dev)
    k = torch.from_numpy(rng.uniform(-math.pi / edge, math.pi / edge, size=(points, 3))).to(dev)
    phase = torch.exp(1j * (k @ shifts.T))
    S, T, B = (torch.einsum("kr,rij->kij", phase, M.to(torch.complex128)) for M in (S_R, T_R, B_R))
    H = T - depth(norb) * (B @ B.mH)
    C0 = torch.from_numpy(rng.normal(0.0, 0.1, size=(points, n, m, 2)) / math.sqrt(2 * m)).to(dev)
    C0 = torch.view_as_complex(C0.contiguous())
    out = []
    for q in range(points):
        Hq, Sq, Tq = (0.5 * (M[q] + M[q].mH) for M in (H, S, T))
        Hq.diagonal().add_(noise)
        out.append((Hq.contiguous(), Sq.contiguous(), Tq.contiguous(), n, C0[q].contiguous()))
    return out


def batch_sizes(case):
    """(units, norb) of every system of a batch: spread between the two ends, kinds in turn."""
    lo, hi, count = case["units_from"], case["units_to"], case["count"]
    units = [round(lo * (hi / lo) ** (i / max(1, count - 1))) for i in range(count)]
    return [(u, (13, 23, 8, 16)[i % 4]) for i, u in enumerate(units)]


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # one small cell per call (64 atoms, minimal basis): m = 256, n = 128; launches and latency count
        {"name": "solve_small", "kind": "solve", "units": 64, "norb": 4, "precision": "mixed", "flavour": "precond"},
        # a mid-size molecular system, odd: 65 molecules, m = 1495, n = 260
        {"name": "solve_medium_odd", "kind": "solve", "units": 65, "norb": 23, "precision": "mixed",
         "flavour": "precond"},
        # the headline size: 512 atoms, m = 6656, n = 1024
        {"name": "solve_large", "kind": "solve", "units": 512, "norb": 13, "precision": "mixed", "flavour": "precond"},
        # the float64 path (reference results), 32 atoms: m = 416, n = 64
        {"name": "solve_fp64", "kind": "solve", "units": 32, "norb": 13, "precision": "fp64", "flavour": "precond"},
        # the S = L L^T flavour: 128 molecules, m = 2944, n = 512
        {"name": "solve_cholesky", "kind": "solve", "units": 128, "norb": 23, "precision": "mixed",
         "flavour": "cholesky"},
        # one step of a self-consistency loop at half filling: m = 2048, n = 1024
        {"name": "scf_step", "kind": "scf", "units": 512, "norb": 4, "precision": "mixed"},
        # the energy inside a torch program, smallest and odd: nine molecules, m = 207, n = 36
        {"name": "autograd_small", "kind": "autograd", "units": 9, "norb": 23},
        # snapshots of uneven size, m from 104 to 1280
        {"name": "batch_uneven", "kind": "batch", "units_from": 8, "units_to": 80, "count": 10},
        # 48 points of a k grid: 48 Hermitian problems, m = 104, n = 16
        {"name": "kpoints", "kind": "kpoints", "points": 48, "units": 8, "norb": 13},
        # one k point in float64
        {"name": "hermitian_fp64", "kind": "hermitian", "units": 8, "norb": 13},
        # inverses of S + T/tau: float64-class at a large size, native at a small one
        {"name": "inverse_sliced", "kind": "inverse", "units": 256, "norb": 13, "sliced": True},
        # the refresh product of the headline size against half of its operators: 1024 x 6656 x 6656
        {"name": "gemm_refresh", "kind": "gemm", "M": 1024, "N": 6656, "K": 6656},
    ]


def log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "scf", "autograd", "batch", "kpoints", "hermitian", "inverse",
                       "gemm", "dgemm"])
    if kind == "solve":
        precision, flavour = rng.choice([("mixed", "precond"), ("mixed", "precond"), ("mixed", "cholesky"),
                                         ("fp64", "precond"), ("fp64", "cholesky")])
        norb = rng.choice([4, 8, 13, 16, 23])
        top = 900 if precision == "fp64" else 2944 if flavour == "cholesky" else {4: 2500, 8: 5000, 23: 3000}.get(norb, 6000)
        return {"kind": kind, "units": max(4, log_int(rng, 100, top) // norb), "norb": norb, "precision": precision,
                "flavour": flavour}
    if kind == "scf":
        norb = rng.choice([4, 8, 13, 23])
        return {"kind": kind, "units": max(8, log_int(rng, 200, 3000 if norb > 4 else 2048) // norb), "norb": norb, "precision": "mixed"}
    if kind == "autograd":
        norb = rng.choice([4, 8, 13, 16, 23])
        return {"kind": kind, "units": max(3, log_int(rng, 60, 500) // norb), "norb": norb}
    if kind == "batch":
        lo = rng.randint(4, 12)
        return {"kind": kind, "units_from": lo, "units_to": lo * rng.randint(2, 8), "count": rng.randint(2, 12)}
    if kind == "kpoints":
        return {"kind": kind, "points": log_int(rng, 4, 96), "units": rng.randint(3, 8),
                "norb": rng.choice([4, 8, 13, 16])}
    if kind == "hermitian":
        return {"kind": kind, "units": log_int(rng, 3, 24), "norb": rng.choice([4, 8, 13, 16])}
    if kind == "inverse":
        norb = rng.choice([4, 8, 13, 16, 23])
        sliced = rng.random() < 0.6
        return {"kind": kind, "units": max(4, log_int(rng, 100, 4000 if sliced else 1500) // norb), "norb": norb,
                "sliced": sliced}
    if kind == "gemm":
        return {"kind": kind, "M": log_int(rng, 32, 2048), "N": log_int(rng, 64, 6656), "K": log_int(rng, 64, 8192)}
    return {"kind": kind, "M": log_int(rng, 16, 512), "N": log_int(rng, 64, 1024), "K": log_int(rng, 64, 1024),
            "transA": rng.random() < 0.3, "transB": rng.random() < 0.5}


def inputs(case, seed, dev):
    """The case's input tensors, from the seed alone."""
    rng = generator(seed)
    kind = case["kind"]
    if kind in ("solve", "scf", "autograd"):
        p = problem(case["units"], case["norb"], rng, dev)
        if kind != "scf":
            return [p]
        # the next step's Hamiltonian: an on-site change of the size of the noise
        H1 = p[0].clone()
        H1.diagonal().add_(torch.from_numpy(rng.normal(0.0, NOISE, size=len(H1))).to(dev))
        return [p, H1]
    if kind == "batch":
        return [problem(u, norb, rng, dev) for u, norb in batch_sizes(case)]
    if kind in ("kpoints", "hermitian"):
        return bloch_problems(case.get("points", 1), case["units"], case["norb"], rng, dev)
    if kind == "inverse":
        _, S, T, _, _ = problem(case["units"], case["norb"], rng, dev)
        return [S + T / TAU]
    # coefficients against operator rows: entries that fall off by orders of magnitude along a row
    M, N, K = case["M"], case["N"], case["K"]
    shape_a = (K, M) if case.get("transA") else (M, K)
    shape_b = (N, K) if kind == "gemm" or case.get("transB") else (K, N)
    g = torch.Generator(device="cpu").manual_seed(int(seed))
    out = []
    for shape in (shape_a, shape_b):
        a = torch.randn(shape, generator=g, dtype=torch.float64).to(dev)
        r = torch.rand(shape, generator=g, dtype=torch.float64).to(dev)
        out.append(a * torch.exp(-6.0 * r))
    return out


def options(case):
    return dict(precision=case["precision"], tol_grad=TOL, cholesky=case.get("flavour") == "cholesky")


def prepare(case, seed):
    kind, dev = case["kind"], torch.device("cuda")
    state = {"case": dict(case), "in": inputs(case, seed, dev)}
    if kind == "scf":  # the loop's context, converged at the previous step's Hamiltonian
        H, S, T, n, C0 = state["in"][0]
        state["solver"] = omm.OMMSolver(H, S, T, n, ETA, TAU, **options(case))
        state["C"] = state["solver"].solve(C0)[0]
    elif kind in ("gemm", "dgemm"):
        state["out"] = torch.empty((case["M"], case["N"]), dtype=torch.float64, device=dev)
    elif kind == "inverse":
        state["out"] = torch.empty_like(state["in"][0])
    elif kind == "autograd":
        H, S, T, n, C0 = state["in"][0]
        state["in"] = [(H.requires_grad_(True), S.requires_grad_(True), T, n, C0)]
    torch.cuda.synchronize()
    return state


def run(state):
    case, given = state["case"], state["in"]
    kind = case["kind"]
    if kind == "solve":
        H, S, T, n, C0 = given[0]
        with omm.OMMSolver(H, S, T, n, ETA, TAU, **options(case)) as s:
            _, E, D, _ = s.solve(C0, want_D=True)
            _, dS = s.backward(want_H=False)
        return {"E": E, "D": D, "dS": dS}
    if kind == "scf":
        s = state["solver"]
        s.update_H(given[1])
        _, E, _, _ = s.solve(state["C"])
        dH, dS = s.backward()
        return {"E": E, "dH": dH, "dS": dS}
    if kind == "autograd":
        H, S, T, n, C0 = given[0]
        E, _ = omm.omm_energy(H, S, T, C0, n, ETA, TAU, tol_grad=TOL)
        dH, dS = torch.autograd.grad(E, (H, S))
        return {"E": E.detach(), "dH": dH, "dS": dS}
    if kind == "batch":
        with omm.OMMBatch([(H, S, T, n, ETA, TAU) for H, S, T, n, _ in given], tol_grad=TOL) as b:
            _, E, _ = b.solve([p[4] for p in given])
            grads = [b.backward(i) for i in range(len(given))]
        return {"E": E, "grads": grads}
    if kind == "kpoints":
        with omm.OMMHermitianBatch([(H, S, T, n, ETA, TAU) for H, S, T, n, _ in given], tol_grad=TOL) as b:
            _, E, _ = b.solve([p[4] for p in given])
            grads = [b.backward(i) for i in range(len(given))]
        return {"E": E, "dH": torch.stack([g[0] for g in grads]), "dS": torch.stack([g[1] for g in grads])}
    if kind == "hermitian":
        H, S, T, n, C0 = given[0]
        with omm.OMMHermitian(H, S, T, n, ETA, TAU, precision="fp64", tol_grad=TOL) as s:
            _, E, _, _ = s.solve(C0)
            dH, dS = s.backward()
        return {"E": E, "dH": dH, "dS": dS}
    if kind == "inverse":
        return steps.spd_inverse(given[0], P=state["out"], sliced=case["sliced"])
    if kind == "gemm":
        return steps.gemm_emu(given[0], given[1], state["out"])
    return steps.dgemm(case["transA"], case["transB"], given[0], given[1], state["out"])


def sizes(case):
    """[(m, n)] of the case's problems, complex ones counted as they are."""
    kind = case["kind"]
    if kind == "batch":
        return [(u * norb, u * occupied(norb)) for u, norb in batch_sizes(case)]
    if kind in ("kpoints", "hermitian"):
        return [(case["units"] * case["norb"], 2 * case["units"])] * case.get("points", 1)
    return [(case["units"] * case["norb"], case["units"] * occupied(case["norb"]))]


def work(case):
    """What one pass cannot do without. A solve: H, S, T and C0 read, two m x m gradients written; the
    inverse, and a line search (its products with P, H and S and with the occupied states) for each of
    thirty steps (ten in a loop's step), fewer than these problems take."""
    kind = case["kind"]
    if kind in ("gemm", "dgemm"):
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 8.0 * (M * K + N * K + M * N), "flops": 2.0 * M * N * K}
    if kind == "inverse":
        m = case["units"] * case["norb"]
        return {"bytes": 16.0 * m * m, "flops": 1.0 * m ** 3}
    z = 4.0 if kind in ("kpoints", "hermitian") else 1.0       # real operations of a complex one
    w = 2.0 if z > 1.0 else 1.0
    count = 10 if kind == "scf" else 30
    total = {"bytes": 0.0, "flops": 0.0}
    for m, n in sizes(case):
        if kind == "scf":
            total["bytes"] += 8.0 * (3 * m * m + n * m)
            total["flops"] += count * (6.0 * m * m * n + 12.0 * m * n * n) + 4.0 * m * m * n
        else:
            total["bytes"] += w * 8.0 * (5 * m * m + n * m)
            total["flops"] += z * (m ** 3 + count * (6.0 * m * m * n + 12.0 * m * n * n) + 4.0 * m * m * n)
    return total


def exact_minimum(H, S, n):
    """E, D and -EDM from the n lowest eigenpairs of H x = eps S x."""
    L = torch.linalg.cholesky(S)
    A = torch.linalg.solve_triangular(L, H, upper=False)
    A = torch.linalg.solve_triangular(L, A.mH.contiguous(), upper=False)
    eps, V = torch.linalg.eigh(0.5 * (A + A.mH))
    X = torch.linalg.solve_triangular(L.mH, V[:, :n].contiguous(), upper=True)
    D = 2.0 * (X @ X.mH)
    EDM = 2.0 * ((X * eps[:n]) @ X.mH)
    return 2.0 * float(eps[:n].sum()), D, -EDM


def exact(case, seed):
    kind, dev = case["kind"], torch.device("cuda")
    if kind in ("gemm", "dgemm"):
        a, b = inputs(case, seed, dev)
        a = a.T if case.get("transA") else a
        b = b.T if kind == "gemm" or case.get("transB") else b
        return a @ b
    if kind == "inverse":
        a = inputs(case, seed, dev)[0]
        return torch.cholesky_inverse(torch.linalg.cholesky(a))
    if max(m for m, _ in sizes(case)) > 4500:  # the eigensolver takes too long
        return None
    given = inputs(case, seed, dev)
    if kind == "scf":
        given = [(given[1],) + given[0][1:]]
    got = [exact_minimum(H, S, n) for H, S, _, n, _ in given]
    if kind == "batch":
        return {"E": np.array([g[0] for g in got]), "grads": [(g[1], g[2]) for g in got]}
    if kind == "kpoints":
        return {"E": np.array([g[0] for g in got]), "dH": torch.stack([g[1] for g in got]),
                "dS": torch.stack([g[2] for g in got])}
    E, D, dS = got[0]
    if kind == "autograd":
        return {"E": torch.tensor(E, dtype=torch.float64), "dH": D, "dS": dS}
    return {"E": E, "D": D, "dS": dS} if kind == "solve" else {"E": E, "dH": D, "dS": dS}
