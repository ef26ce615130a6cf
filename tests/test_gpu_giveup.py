"""The inner solver's bounded waits when a sum never comes: tests/kmix_giveup_check.cu,
which holds the library's kernel with a limit of 5 ms, compiled and run."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_missing_sums(tmp_path):
    from paper_2104_04609_gb300 import build

    exe = tmp_path / "kmix_giveup_check"
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, os.path.join(HERE, "kmix_giveup_check.cu"), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.startswith("ok "), r.stdout
    print(r.stdout)
