"""Calls of which one kernel launch is refused: the call returns an error, and
the calls after it give what they give without it.

The refusal is made on the host, by a stand-in for the runtime's launch
functions that is linked with the library's objects (tests/launch_fault.cu) into
a copy of the package; each case runs it in a process of its own and compares
with a scene that saw no refusal."""

import glob
import os
import shutil
import subprocess
import sys

import pytest

from paper_1708_00783_gb300 import build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

COMMON = r"""
import ctypes, numpy as np, torch
import paper_1708_00783_gb300 as itm
from synth import tiny_workload
from tests.test_gpu_mesh import canonical, gpu_mesh
assert itm.__file__.startswith(%(pkg)r), itm.__file__
lib = ctypes.CDLL(itm.LIB_PATH)
w = tiny_workload(n_frames=10)
i = w.intr
ci = itm.make_intrinsics(i.width, i.height, i.fx, i.fy, i.cx, i.cy)
depth = lambda k: torch.from_numpy(w.frame(k).depth).cuda()
pose = lambda k: w.frame(k).T_wc
maps = lambda: [torch.full((i.height, i.width, 4), 7.0, device="cuda") for _ in range(2)]

def refused(n, call):
    "call with its n-th launch refused"
    torch.cuda.synchronize()
    lib.launch_fault_in(n)
    try:
        call()
    except Exception as e:
        assert lib.launch_fault_left() == 0, "launch not reached"
        torch.cuda.synchronize()
        return
    raise AssertionError("no error")

def same(a, b):
    torch.cuda.synchronize()
    return all(torch.equal(x, y) for x, y in zip(a, b))

def volume(s):
    c, F, W = s.export()
    o = np.lexsort(c.T[::-1])
    return c[o], F[o], W[o]

def same_volume(a, b):
    return all(np.array_equal(x, y) for x, y in zip(volume(a), volume(b)))
"""


@pytest.fixture(scope="module")
def package(tmp_path_factory):
    """A copy of the package whose library can be told to refuse a launch."""
    d = tmp_path_factory.mktemp("launch_fault")
    pkg = d / "paper_1708_00783_gb300"
    (pkg / "_lib").mkdir(parents=True)
    for f in glob.glob(os.path.join(build.HERE, "*.py")):
        shutil.copy(f, pkg)
    objs = [os.path.join(build.OBJ_DIR, s.replace(".cu", ".o")) for s in sorted(build.SOURCES)]
    if not all(map(os.path.exists, objs)):
        build.build(force=True)
    wraps = [x for s in ("cudaLaunchKernelExC", "__cudaLaunchKernel", "cudaGetLastError") for x in ("-Xlinker", "--wrap=" + s)]
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    os.path.join(HERE, "launch_fault.cu"), *objs, *wraps, "-o", str(pkg / "_lib" / "libitm.so")],
                   check=True, capture_output=True, text=True)
    return d


def run(package, script):
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([str(package), ROOT, os.environ.get("PYTHONPATH", "")]))
    r = subprocess.run([sys.executable, "-c", COMMON % {"pkg": str(package)} + script], cwd=str(package), env=env,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.stdout[-2000:], r.stderr[-3000:])


def test_raycast(package):
    """The march refused, then the finish (beside a search range of another pose): the next raycasts are whole."""
    run(package, r"""
g = itm.Scene(**w.params)
for k in range(3):
    g.process(depth(k), ci, pose(k), *maps())
want = {}
for k in (2, 9):
    want[k] = maps()
    g.raycast(ci, pose(k), *want[k])
torch.cuda.synchronize()
# a raycast whose search range is there launches march and finish, another the range first
for n, before, k in ((1, 9, 9), (2, 9, 9), (2, 9, 2), (3, 9, 2), (2, 2, 2), (2, 2, 9)):
    g.raycast(ci, pose(before), *maps())
    refused(n, lambda: g.raycast(ci, pose(k), *maps()))
    for again in (before, 2, 9, 2):
        got = maps()
        g.raycast(ci, pose(again), *got)
        assert same(got, want[again]), (n, before, k, again)
""")
