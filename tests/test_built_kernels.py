"""Batched plane kernels are built only where a batch's members (at most BATCH_MAX_TILES tiles) can
take them: FP32 pairs of degree 1, and Cartesian ones of degrees 1 to 3."""
import re
import shutil
import subprocess

import pytest

from paper_2609_04534_gb300 import build


def test_batched_plane_kernels_are_those_a_request_can_reach():
    if not shutil.which("nm"):
        pytest.skip("nm not found")
    names = subprocess.run(["nm", "-C", build.build()], capture_output=True, text=True, timeout=300).stdout
    general = set(re.findall(r"apply_general_plane_batch<(\w[\w:]*), ([\w:]+), (\d+),", names))
    cartesian = set(re.findall(r"apply_cartesian_plane_batch<(\w[\w:]*), ([\w:]+), (\d+),", names))
    assert general == {("float", "mf::f2", "2")}, general
    assert cartesian == {("float", "mf::f2", n) for n in "234"}, cartesian
