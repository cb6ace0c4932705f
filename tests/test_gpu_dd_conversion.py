"""The double-float -> double conversion as the device does it (mf_dd.cuh) equals the host's
integer form over normalised pairs and the edge cases (tests/dd_device_check.cu, compiled here)."""
import os
import shutil
import subprocess

import pytest

from paper_2609_04534_gb300 import build

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_device_conversion_equals_the_host_form(tmp_path):
    nvcc = build.nvcc()
    if not shutil.which(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "dd_device_check"
    r = subprocess.run([nvcc, *build.ARCH, "-O2", "-std=c++17", "-I", build.CSRC, "-o", str(exe),
                        os.path.join(ROOT, "tests", "dd_device_check.cu")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("ok"), r.stdout + r.stderr
