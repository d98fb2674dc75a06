"""Places of the brick table along a walk: blocks enter and leave, bricks meet at
places, and a place is marked or taken only as long as a block counts on it
(tests/brick_leave_check.cu)."""

import os
import subprocess

import pytest

from paper_1708_00783_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.gpu
def test_places_are_given_back(tmp_path):
    exe = str(tmp_path / "brick_leave_check")
    subprocess.check_call([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I",
                           build.INCLUDE, "-I", build.CSRC, os.path.join(HERE, "brick_leave_check.cu"), "-o", exe])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
