"""Compiles the C++ and CUDA programs of tests/native."""
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
PKG = os.path.join(os.path.dirname(HERE), "paper_1312_1549_gb300")


def compile_program(name, out, *flags):
    """out/<stem> from tests/native/<name>: nvcc for .cu, g++ for .cpp."""
    exe = os.path.join(str(out), os.path.splitext(name)[0])
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    cxx = [nvcc] if name.endswith(".cu") else ["g++", "-Wno-unknown-pragmas"]
    subprocess.run(cxx + ["-std=c++17", "-O1", "-I", os.path.join(PKG, "csrc"), "-I", os.path.join(HERE, "native"),
                          os.path.join(HERE, "native", name), "-o", exe, *flags], check=True)
    return exe


def run_program(exe, *args, timeout=300):
    r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=timeout)
    assert r.returncode == 0, r.stdout[-4000:] + r.stderr[-4000:]
    return r.stdout
