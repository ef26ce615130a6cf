"""The mixed inner solver's matrix entries: tests/kmix_entry_check.cu, which holds
the library's kernel, compiled and run."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def test_cancelling_entries(tmp_path):
    from paper_2104_04609_gb300 import build

    exe = tmp_path / "kmix_entry_check"
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, os.path.join(HERE, "kmix_entry_check.cu"), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.endswith("ok\n"), r.stdout
