"""Host check of the block-wide bounded wait (csrc/bounded_wait.cuh) and of the
inner solver's status words, compiled with g++ and run with threads; no GPU."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_INC = os.environ.get("CUDA_HOME", "/usr/local/cuda") + "/include"


def test_bounded_wait(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers not available")
    exe = tmp_path / "bounded_wait_check"
    subprocess.run([gxx, "-O2", "-std=c++17", "-pthread", "-I" + CUDA_INC,
                    os.path.join(HERE, "bounded_wait_check.cpp"), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("ok "), r.stdout
