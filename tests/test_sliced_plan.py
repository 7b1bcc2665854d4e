"""How sliced products are shared among the SMs, followed on the host (CPU)."""
from native_build import compile_program, run_program


def test_every_stage_has_one_worker_and_every_share_a_length(tmp_path):
    run_program(compile_program("sliced_plan.cu", tmp_path))
