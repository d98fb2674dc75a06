"""The brick table's addressing, on the CPU: tests/brick_check.cu compiled for the
host enters random blocks and reads every neighbourhood back."""

import os
import subprocess

import pytest

from paper_1708_00783_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def test_neighbourhoods_read_back(tmp_path):
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = str(tmp_path / "brick_check")
    subprocess.run([cc, *build.ARCH, "-O2", "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC,
                    "--expt-relaxed-constexpr", os.path.join(HERE, "brick_check.cu"), "-o", exe], check=True,
                   capture_output=True, text=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout
