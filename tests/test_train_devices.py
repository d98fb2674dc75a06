"""The training step asks for its shared memory on every device it is used on
(tests/train_devices_check.cu, the library's objects with a stand-in for the
runtime; no GPU)."""

import os
import subprocess

import pytest

from paper_1708_00783_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
WRAPPED = ["cudaGetDevice", "cudaDeviceGetAttribute", "cudaOccupancyMaxActiveBlocksPerMultiprocessor",
           "cudaFuncSetAttribute", "__cudaGetKernel", "__cudaLaunchKernel", "cudaGetLastError"]


def test_step_on_two_devices(tmp_path):
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    objs = [os.path.join(build.OBJ_DIR, s.replace(".cu", ".o")) for s in sorted(build.SOURCES)]
    if not all(map(os.path.exists, objs)):
        build.build(force=True)
    exe = str(tmp_path / "train_devices_check")
    subprocess.run([cc, *build.ARCH, "-O2", "-std=c++17", "-I", build.INCLUDE,
                    os.path.join(HERE, "train_devices_check.cu"), *objs, "-ldl", "-lpthread",
                    *[x for s in WRAPPED for x in ("-Xlinker", "--wrap=" + s)], "-o", exe],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120, check=True).stdout.split()
    assert out == ["0"] * 6, out
