"""Host check of the GEMM's MMA shapes (csrc/umma_shape.cuh), compiled with g++
and run; no GPU."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_mma_shapes(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "umma_shape_check"
    subprocess.run([gxx, "-O1", "-std=c++17", "-Wall", "-Werror", os.path.join(HERE, "umma_shape_check.cpp"), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout == "ok 16\n", r.stdout
