"""The float64 leaf of the Cholesky inverses on the host, its warps in different orders between the block
barriers: the results may not depend on how far another warp has come (CPU)."""
from native_build import compile_program, run_program


def test_leaf_does_not_depend_on_the_warp_order(tmp_path):
    run_program(compile_program("leaf_f64.cpp", tmp_path))
