"""The workspaces of the tensor-core inverses."""
import ctypes as ct
import os

import pytest

from native_build import compile_program, run_program

GPU = pytest.mark.gpu


def test_workspace_sizes():
    """Without the lane that runs ahead, at most what the inverse took before it had one (2.3 m^2 float64 and 20 m^2
    bytes of slices beside the caller's m^2, and 430 MB of sums); the split form takes its three bf16 pairs only."""
    from paper_1312_1549_gb300 import build
    lib = ct.CDLL(build.build())
    size = lib._ZN3omm34spd_inverse_sliced_workspace_bytesEiib
    size.restype, size.argtypes = ct.c_size_t, [ct.c_int, ct.c_int, ct.c_bool]
    for m in (2048, 3328, 6656, 20000, 54321):
        assert size(m, 10, False) <= 38.4 * m * m + 430e6
        assert size(m, 10, True) <= (14 + 32) * (m + 300.0) ** 2 + 250e6
        assert size(m, 1, True) == size(m, 1, False) <= 12 * (m + 64.0) ** 2 + 256


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_1312_1549_gb300 import build
    lib = build.build()
    return compile_program("inverse_workspace.cu", tmp_path_factory.mktemp("native"), *build.ARCH, lib, "-Xlinker",
                           "-rpath=" + os.path.dirname(lib))


@GPU
@pytest.mark.parametrize("m", [65, 200, 500, 1100])
@pytest.mark.parametrize("slices", [1, 5, 10])
def test_same_result_without_the_lane_that_runs_ahead(program, m, slices):
    run_program(program, m, slices)
