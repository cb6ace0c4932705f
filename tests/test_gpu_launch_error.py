"""A kernel launch that the runtime refuses is reported by the call that made it, and only there
(tests/launch_error_check.cu, compiled here)."""
import os
import shutil
import subprocess

import pytest

from paper_2609_04534_gb300 import build

pytestmark = pytest.mark.gpu


def test_a_refused_launch_leaves_no_error_behind(tmp_path):
    nvcc = build.nvcc()
    if not shutil.which(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "launch_error_check"
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "launch_error_check.cu")
    r = subprocess.run([nvcc, *build.ARCH, "-O2", "-std=c++17", "-I", build.CSRC, "-o", str(exe), src],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
