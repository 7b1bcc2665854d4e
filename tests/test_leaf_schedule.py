"""The float64 leaf of the Cholesky inverses on the host, its warps in different orders between the block
barriers: the results may not depend on how far another warp has come (CPU)."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_1312_1549_gb300", "csrc")


def test_leaf_does_not_depend_on_the_warp_order(tmp_path):
    exe = str(tmp_path / "leaf")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wno-unknown-pragmas", "-I", CSRC, "-I", os.path.join(HERE, "native"),
                    os.path.join(HERE, "native", "leaf_f64.cpp"), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
