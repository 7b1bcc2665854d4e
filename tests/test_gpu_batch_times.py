"""The recompute times that the instances of a batch report are shares of the batch's time."""
import numpy as np
import pytest
import torch

from test_gpu_batch_states import dev, pencil

pytestmark = pytest.mark.gpu


def test_grouped_recomputes_are_not_counted_for_each_instance():
    from paper_1312_1549_gb300 import OMMBatch
    rng = np.random.default_rng(8)
    count, m, n = 96, 48, 12
    ps = [pencil(m, n, rng) for _ in range(count)]
    with OMMBatch([(dev(H), dev(S), dev(np.eye(m)), n, 0.0, 5.0) for H, S, _, _ in ps]) as b:
        _, _, infos = b.solve([dev(p[3]) for p in ps])
    total = sum(i["ms_refine"] for i in infos)
    assert 0.0 < total <= infos[0]["ms_batch"]
    assert all(i["ms_certify"] > 0.0 for i in infos)
