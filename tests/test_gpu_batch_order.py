"""A batch reads its inputs after what is queued on its stream."""
import numpy as np
import pytest
import torch

from test_gpu_batch_states import dev, pencil

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_inputs_still_being_written(precision):
    from paper_1312_1549_gb300 import OMMBatch
    rng = np.random.default_rng(21)
    m, n = 64, 16
    ps = [pencil(m, n, rng) for _ in range(3)]
    T = dev(np.eye(m))
    ready = [[dev(H), dev(S)] for H, S, _, _ in ps]
    inputs = [[torch.eye(m, device="cuda", dtype=torch.float64).neg_() for _ in range(2)] for _ in ps]  # not even definite
    C0 = [dev(p[3]) for p in ps]
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        torch.cuda._sleep(40_000_000)  # some 20 ms
        for dst, src in zip(inputs, ready):
            for d, s in zip(dst, src):
                d.copy_(s)
    with OMMBatch([(H, S, T, n, 0.0, 5.0) for H, S in inputs], precision=precision, stream=st) as b:
        _, E, _ = b.solve(C0)
    for e, p in zip(E, ps):
        assert abs(e - p[2]) <= 1e-9 * abs(p[2])
