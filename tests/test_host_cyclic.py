"""Host-side check of the one-range activity test that the scan and
asse_estimate use (Algorithms 1 and 2 on packed words), against the algorithms
per value for every k, k', ACT and value, and on words of every field width.
Built with the host compiler, no GPU needed."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
BUILD = os.path.join(ROOT, "tests", "host", "_build")


def test_cyclic_ranges_match_the_algorithms():
    cxx = shutil.which("g++")
    cuda_inc = "/usr/local/cuda/include"
    if cxx is None or not os.path.exists(os.path.join(cuda_inc, "vector_types.h")):
        pytest.skip("needs g++ and the CUDA headers")
    os.makedirs(BUILD, exist_ok=True)
    exe = os.path.join(BUILD, "cyclic")
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_1807_01527_gb300", "csrc"), "-I", cuda_inc,
                    os.path.join(ROOT, "tests", "host", "cyclic.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.split()[-1] == "ok", out.stdout
