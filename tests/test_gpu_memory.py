"""Device memory that contexts hold and that calls give back, each in a fresh process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = """
import torch
import paper_1312_1549_gb300 as omm
from paper_1312_1549_gb300 import solver as steps

def taken(start=[None]):   # bytes of the device taken since the first call
    free = torch.cuda.mem_get_info()[0]
    if start[0] is None:
        start[0] = free
    return start[0] - free

def system(m, n):
    g = torch.Generator(device="cuda").manual_seed(m)
    X = torch.randn((m, m), generator=g, device="cuda", dtype=torch.float64) / m ** 0.5
    S = torch.eye(m, device="cuda", dtype=torch.float64) + 0.1 * (X + X.T)
    d = torch.linspace(-3.0, -2.0, m, device="cuda", dtype=torch.float64)
    d[n:] += 5.0
    C0 = torch.randn((n, m), generator=g, device="cuda", dtype=torch.float64) * (0.1 / m ** 0.5)
    return (torch.diag(d) + 0.05 * (X + X.T)).contiguous(), S.contiguous(), C0
"""


def run(code):
    r = subprocess.run([sys.executable, "-c", PRELUDE + code], cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]


def test_contexts_hold_no_slabs():
    """24 contexts with float64-class refreshes take less than 24 slabs of sliced products alone would (80 MB each);
    a solve, its density and its gradients still run in all of them."""
    run("""
m, n = 512, 256
H, S, C0 = system(m, n)
omm.OMMSolver(H, S, S, n, 4.5, 5.0, precision="mixed").close()
taken()
solvers = [omm.OMMSolver(H, S, S, n, 4.5, 5.0, precision="mixed") for _ in range(24)]
assert taken() < 24 * 80e6, taken()
ref = None
for s in solvers[::8]:
    C, E, D, info = s.solve(C0, want_D=True)
    dH, dS = s.backward()
    assert torch.equal(D, dH)
    ref = D if ref is None else ref
    assert torch.equal(D, ref)
""")


def test_scratch_of_a_call_is_given_back():
    """The float64-class inverse of m = 9472 takes more than 4 GB of scratch; at most 2 GiB of it stay reserved after
    the call (allowing for the driver's 64 MiB), and nothing after release_unused."""
    run("""
m = 9472
A = torch.eye(m, device="cuda", dtype=torch.float64)
P = torch.empty_like(A)
small = torch.eye(64, device="cuda", dtype=torch.float64)
steps.spd_inverse(small, sliced=True)
steps.release_unused()
torch.cuda.synchronize()
taken()
steps.spd_inverse(A, P, sliced=True)
assert taken() <= (2 << 30) + (64 << 20), taken()
steps.release_unused()
assert taken() <= 64 << 20, taken()
assert torch.equal(P, A)
""")
