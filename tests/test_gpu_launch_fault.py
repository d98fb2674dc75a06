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


# what follows an allocation of which the commit ran and the visible-list pass did not
AFTER = {
    "allocate": r"""
for s in (g, o):
    s.process(depth(9), ci, pose(9), *maps())
""",
    "raycast": r"""
m = [maps(), maps()]
for s, x in ((g, m[0]), (o, m[1])):
    s.raycast(ci, pose(9), *x)
assert same(*m)
""",
    "mesh": r"""
a, b = gpu_mesh(itm, g), gpu_mesh(itm, o)
assert len(a) > 0 and np.array_equal(canonical(a), canonical(b))
""",
    "combined": r"""
m = [maps(), maps()]
eye = np.eye(4, dtype=np.float32)[None]
for s, x in ((g, m[0]), (o, m[1])):
    itm.itm_raycast_combined([s.handle], eye, ci, pose(9), *x)
assert same(*m)
""",
    "batch": r"""
b = itm.itm_batch_create(1)
m = [maps(), maps()]
for s, x in ((g, m[0]), (o, m[1])):
    itm.itm_batch_run(b, [(s.handle, depth(9), ci, pose(9), x[0], x[1])])
assert same(*m)
""",
    "swap_out": r"""
for s in (g, o):
    s.swap_out()
    for k in (9, 0, 5, 9):
        s.allocate(depth(k), ci, pose(k))
        s.swap_in()
        s.integrate(depth(k), ci, pose(k))
        s.swap_out()
assert g.swap_counters()["moved_out"] == o.swap_counters()["moved_out"] > 0
""",
    "reset": r"""
for s in (g, o):
    s.reset()
    s.process(depth(5), ci, pose(5), *maps())
""",
    "import": r"""
v = g.export()
for s in (g, o):
    s.import_blocks(*v)
""",
}


@pytest.mark.parametrize("then", sorted(AFTER))
def test_allocation_without_its_visible_list(package, then):
    """The blocks of the refused frame are found by whatever comes next, and no key is entered twice."""
    run(package, r"""
g, o = itm.Scene(**w.params), itm.Scene(**w.params)
if %r == "swap_out":
    for s in (g, o):
        s.swap_enable(4096, 0)
for s in (g, o):
    for k in (0, 1):
        s.process(depth(k), ci, pose(k), *maps())
before = g.stats()["allocated_blocks"]
refused(3, lambda: g.allocate(depth(9), ci, pose(9)))
o.allocate(depth(9), ci, pose(9))
assert g.stats()["allocated_blocks"] > before + 100
""" % then + AFTER[then] + r"""
assert g.status() == o.status() == 0
assert same_volume(g, o)
for k in (9, 5, 0):
    for s in (g, o):
        s.allocate(depth(k), ci, pose(k))
        if %r == "swap_out":
            s.swap_in()
        s.integrate(depth(k), ci, pose(k))
    m = [maps(), maps()]
    g.raycast(ci, pose(k), *m[0])
    o.raycast(ci, pose(k), *m[1])
    assert same(*m), k
assert same_volume(g, o) and g.status() == o.status() == 0
""" % then)


@pytest.mark.parametrize("n", [1, 2])
def test_allocation_refused_before(package, n):
    """The enumeration or the commit refused: the frame can be repeated."""
    run(package, r"""
g, o = itm.Scene(**w.params), itm.Scene(**w.params)
for s in (g, o):
    s.process(depth(0), ci, pose(0), *maps())
refused(%d, lambda: g.allocate(depth(9), ci, pose(9)))
for k in (9, 5):
    m = [maps(), maps()]
    g.process(depth(k), ci, pose(k), *m[0])
    o.process(depth(k), ci, pose(k), *m[1])
    assert same(*m), k
    assert g.stats()["allocated_blocks"] == o.stats()["allocated_blocks"]
assert same_volume(g, o) and g.status() == o.status() == 0
""" % n)


def test_import_and_reset(package):
    """Every launch of an import and of a reset refused in turn, then done again."""
    run(package, r"""
g, o = itm.Scene(**w.params), itm.Scene(**w.params)
for s in (g, o):
    s.process(depth(0), ci, pose(0), *maps())
v = o.export()
for n in (1, 2, 3, 4):
    refused(n, lambda: g.import_blocks(*v))
    for _ in range(2):  # what the failed one left is not the volume: import again
        g.import_blocks(*v)
    m = [maps(), maps()]
    g.raycast(ci, pose(0), *m[0])
    o.raycast(ci, pose(0), *m[1])
    assert same(*m) and same_volume(g, o), n
for n in (1, 2, 3):
    refused(n, g.reset)
    g.reset()
    m = [maps(), maps()]
    g.process(depth(0), ci, pose(0), *m[0])
    o.reset()
    o.process(depth(0), ci, pose(0), *m[1])
    assert same(*m) and same_volume(g, o), n
""")


@pytest.mark.parametrize("n", range(1, 10))
def test_batch(package, n):
    """Each launch of a batch without a captured graph refused in turn, then the frame once more."""
    run(package, r"""
scenes = []
for p in (w.params, dict(w.params, num_buckets=1 << 8, num_excess=1 << 13)):
    scenes.append((itm.Scene(**p), itm.Scene(**p)))
b = itm.itm_batch_create(4)
itm.itm_batch_set_graph(b, 0)

def frame(side, k):
    m = [maps() for _ in scenes]
    items = [(s[side].handle, depth(k), ci, pose(k), v, n) for s, (v, n) in zip(scenes, m)]
    itm.itm_batch_run(b, items)
    return m

for k in (0, 1):
    frame(0, k), frame(1, k)
refused(%d, lambda: frame(0, 9))
if %d <= 6:  # stages: begin, enumerate, commit, overflow, visible, integrate, range, march, finish
    frame(0, 9)
frame(1, 9)
for k in (5, 0):
    for x, y in zip(frame(0, k), frame(1, k)):
        assert same(x, y), k
for g, o in scenes:
    assert g.status() == o.status() == 0
    assert g.stats()["allocated_blocks"] == len(g.export(False)[0])
    assert same_volume(g, o)
""" % (n, n))


@pytest.mark.parametrize("n", range(1, 7))
def test_swap_out(package, n):
    """Each launch of a swap-out refused in turn (scan, count, select, move, the two of the compaction): up to the
    move every block stays, after it those that moved are not found in device memory."""
    run(package, r"""
g, o = itm.Scene(**w.params), itm.Scene(**w.params)
for s in (g, o):
    s.swap_enable(1 << 14, 0)
    for k in (0, 1, 2):
        s.process(depth(k), ci, pose(k), *maps())
refused(%d, g.swap_out)
if %d > 4:
    o.swap_out()
for k in (9, 5, 0):
    m = [maps(), maps()]
    for s, x in ((g, m[0]), (o, m[1])):
        s.raycast(ci, pose(0), *x)
    assert same(*m), k
    for s in (g, o):
        s.allocate(depth(k), ci, pose(k))
        s.swap_in()
        s.integrate(depth(k), ci, pose(k))
    assert same_volume(g, o), k
assert g.status() == o.status() == 0
for s in (g, o):
    s.swap_out()
    s.process(depth(3), ci, pose(3), *maps())
m = [maps(), maps()]
g.raycast(ci, pose(3), *m[0])
o.raycast(ci, pose(3), *m[1])
assert same(*m) and same_volume(g, o) and g.status() == o.status() == 0
""" % (n, n))
