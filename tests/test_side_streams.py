"""The side streams of the inverses when a call fails midway, on a fake CUDA runtime (CPU)."""
import os
import shutil

from native_build import compile_program, run_program


def test_no_work_goes_on_that_nobody_waits_for(tmp_path):
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    run_program(compile_program("side_streams.cpp", tmp_path, "-I", include))
