"""The tracker's step kernel where its threads take more than one pass of pixels
(a full grid of two CTAs per SM, eight pixels per thread, and images just
beyond it), and the reciprocal its solve takes (tests/rcp_double_check.cu).

Sums: the bound of test_gpu_track.py, 2e-6 of the magnitude of the terms: here a
thread adds up to 16 products in float and the warp five more times, 21
roundings of 2^-24, 1.3e-6."""

import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1708_00783_gb300 import build
from tests.test_gpu_track_steps import _case
from tests.test_oracle_track_pins import exp_pose

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.mark.parametrize("dw,dh", [(-1, 0), (0, 0), (1, 0), (0, 1), (8, 8)])
def test_sums_around_a_second_pass(dw, dh):
    """A full pass of the full grid is 8 SMs x 512 pixels; a column less, and a column or a row more."""
    import torch
    import paper_1708_00783_gb300 as itm
    W, H = 8 * torch.cuda.get_device_properties(0).multi_processor_count + dw, 512 + dh
    intr, d, V, N = _case(W, H)
    ci = itm.make_intrinsics(W, H, intr.fx, intr.fy, intr.cx, intr.cy)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    Tref = np.eye(4, dtype=np.float32)
    Tg = exp_pose(np.array([0.01, -0.02, 0.01, 0.01, 0.0, 0.01]), Tref)
    work = torch.zeros(itm.ITM_ICP_WORK_DOUBLES, dtype=torch.float64, device="cuda")
    itm.itm_icp_reduce(dev(d), ci, Tg, dev(V), dev(N), ci, Tref, 0.3, work)
    torch.cuda.synchronize()
    g = work[:29].cpu().numpy()
    o, a = oracle.icp_reduce(d, intr.as_array(), Tg, V, N, intr.as_array(), Tref, 0.3)
    assert g[28] == o[28] and o[28] >= 1
    assert np.all(np.abs(g[:28] - o[:28]) <= 2e-6 * np.asarray(a)[:28] + 1e-12)


def test_double_reciprocal(tmp_path):
    objs = [os.path.join(build.OBJ_DIR, s.replace(".cu", ".o")) for s in sorted(build.SOURCES) if s != "itm_track.cu"]
    if not all(map(os.path.exists, objs)):
        build.build(force=True)
    exe = str(tmp_path / "rcp_double_check")
    subprocess.check_call([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-fmad=false", "--expt-relaxed-constexpr",
                           "-I", build.INCLUDE, "-I", build.CSRC, os.path.join(HERE, "rcp_double_check.cu"), *objs,
                           "-ldl", "-lpthread", "-o", exe])
    out = list(map(int, subprocess.run([exe], capture_output=True, text=True, timeout=300, check=True).stdout.split()))
    assert out[0] <= 1 and out[1] == 0, out
