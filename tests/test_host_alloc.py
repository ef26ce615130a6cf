"""Host checks of what a failed device allocation leaves behind, compiled with
g++ against the library's headers and an allocator that fails on demand; no
GPU."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA_INC = os.environ.get("CUDA_HOME", "/usr/local/cuda") + "/include"


def _run(tmp_path, name):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers not available")
    exe = tmp_path / name
    subprocess.run([gxx, "-O1", "-std=c++17", "-I" + CUDA_INC, os.path.join(HERE, name + ".cpp"), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("ok "), r.stdout


def test_buffer_after_failed_allocation(tmp_path):
    _run(tmp_path, "dbuf_check")
