"""The lanes of a warp of the raycast's first phase stop together: the length of
the slow list, which other warps add to meanwhile, is read once per warp
(tests/march_stop_check.cu)."""

import os
import subprocess

import pytest

from paper_1708_00783_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.gpu
def test_lanes_of_a_warp_stop_together(tmp_path):
    exe = str(tmp_path / "march_stop_check")
    subprocess.check_call([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-fmad=false", "--expt-relaxed-constexpr",
                           "-I", build.INCLUDE, "-I", build.CSRC, os.path.join(HERE, "march_stop_check.cu"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120, check=True).stdout.split()
    apart, stopped, went_on = map(int, out)
    assert apart == 0 and stopped > 0 and went_on > 0, out
