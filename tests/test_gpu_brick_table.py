"""The brick table after everything that moves blocks: allocation in any order,
hash chains, batches, swap-out and return, import, reset, holes in the map, and
bricks that share a place of the table.

The raycast and the mesh look blocks up in the brick table.  A volume that is
exported and imported into a fresh scene is entered from scratch, so the two
scenes must give the same maps bit for bit and the same triangles; volumes with
holes, and two views of the tiny scene that lie some 43 bricks apart (with the
smallest table, every brick of one has the place of its twin in the other, so
lookups go to the hash table), are compared with the oracle (the bars of
parity_util.py)."""

import dataclasses

import numpy as np
import pytest

import oracle
from synth import tiny_workload
from tests.parity_util import compare_raycast, compare_volumes
from tests.test_gpu_mesh import canonical, gpu_mesh
from tests.test_gpu_swap import run as run_swapping

pytestmark = pytest.mark.gpu

# bricks this far apart have the same place in the smallest table (and the views do not touch)
TWIN = np.array([43, 1, -4])


@pytest.fixture(scope="module")
def itm():
    import torch
    assert torch.cuda.is_available()
    import paper_1708_00783_gb300 as m
    return m


class Case:
    def __init__(self, itm, **params):
        self.itm, self.w = itm, tiny_workload(n_frames=10)
        self.params = dict(self.w.params, **params)
        i = self.w.intr
        self.ci = itm.make_intrinsics(i.width, i.height, i.fx, i.fy, i.cx, i.cy)
        self.scene = itm.Scene(**self.params)

    def depth(self, k):
        import torch
        return torch.from_numpy(self.w.frame(k).depth).cuda()

    def maps(self):
        import torch
        v = torch.full((self.w.intr.height, self.w.intr.width, 4), 7.0, device="cuda")
        return v, torch.full_like(v, 7.0)

    def process(self, k, scene=None):
        (scene or self.scene).process(self.depth(k), self.ci, self.w.frame(k).T_wc, *self.maps())

    def check_against_import(self, poses=(0, 5, 9), mesh=True):
        import torch
        fresh = self.itm.Scene(**dict(self.params, num_buckets=1 << 14, num_excess=1 << 14))
        fresh.import_blocks(*self.scene.export())
        for k in poses:
            a, b = self.maps(), self.maps()
            T = self.w.frame(k).T_wc
            self.scene.raycast(self.ci, T, *a)
            fresh.raycast(self.ci, T, *b)
            torch.cuda.synchronize()
            assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1]), k
        if mesh:
            ta, tb = gpu_mesh(self.itm, self.scene), gpu_mesh(self.itm, fresh)
            assert len(ta) > 0 and np.array_equal(canonical(ta), canonical(tb))
        assert self.scene.status() == 0


@pytest.mark.parametrize("buckets,excess", [(1 << 16, 1 << 14), (1 << 8, 1 << 13)])
def test_growth_in_any_order(itm, buckets, excess):
    """Blocks that come before and after their neighbours, in wide tables and in long chains."""
    c = Case(itm, num_buckets=buckets, num_excess=excess, num_blocks=1 << 13)
    for k in (5, 0, 9, 3, 7, 1):
        c.process(k)
        c.check_against_import(poses=(k,), mesh=k == 1)
    c.check_against_import()


def test_batch_and_single_calls_in_turn(itm):
    c = Case(itm, num_blocks=1 << 13)
    b = itm.itm_batch_create(2)
    for j, k in enumerate((4, 0, 9, 6)):
        if j & 1:
            v, n = c.maps()
            itm.itm_batch_run(b, [(c.scene.handle, c.depth(k), c.ci, c.w.frame(k).T_wc, v, n)])
        else:
            c.process(k)
    c.check_against_import()
    itm.itm_batch_destroy(b)


@pytest.mark.parametrize("K,idle", [(64, 1), (4096, 0)])
def test_swapped_out_and_back(itm, K, idle):
    """Blocks leave, others take their indices, they return elsewhere."""
    c = Case(itm, num_blocks=1 << 13)
    c.scene.swap_enable(K, idle)
    for k in (0, 9, 0, 5, 9, 1, 0, 8, 4):
        T = c.w.frame(k).T_wc
        d = c.depth(k)
        c.scene.allocate(d, c.ci, T)
        c.scene.swap_in()
        c.scene.integrate(d, c.ci, T)
        c.check_against_import(poses=(k, 9 - k), mesh=False)
        c.scene.swap_out()
        c.check_against_import(poses=(k, 9 - k), mesh=False)
    n = c.scene.swap_counters()
    assert n["moved_out"] > 200 and n["moved_in"] > 50


def test_reset_and_again(itm):
    c = Case(itm, num_blocks=1 << 13)
    c.process(0)
    c.scene.reset()
    c.process(9)
    c.process(5)
    c.check_against_import()


@pytest.mark.parametrize("keep", [0.5, 0.9])
def test_holes_in_the_map(itm, keep):
    """A random share of a fused map's blocks: stencils that start in a missing block, and stencils with missing blocks."""
    import torch
    c = Case(itm, num_blocks=1 << 13)
    for k in (0, 5, 9):
        c.process(k)
    coords, sdf, wgt = c.scene.export()
    sel = np.random.default_rng(3).uniform(size=len(coords)) < keep
    holed, o = itm.Scene(**c.params), oracle.Scene(**c.params)
    holed.import_blocks(coords[sel], sdf[sel], wgt[sel])
    for b, F, W in zip(coords[sel], sdf[sel], wgt[sel]):
        o.set_block(b, F, W)
    i = c.w.intr
    for k in (0, 9):
        T = c.w.frame(k).T_wc
        v, n = c.maps()
        holed.raycast(c.ci, T, v, n)
        torch.cuda.synchronize()
        vo, no = o.raycast(i.width, i.height, i.as_array(), T)
        rep = compare_raycast(v.cpu().numpy(), n.cpu().numpy(), vo, no, T)
        assert rep["hits"] > 1000
    assert np.array_equal(canonical(gpu_mesh(itm, holed)), canonical(o.mesh()))


class Twins:
    """Frame 2 k of the tiny workload's view k, frame 2 k + 1 its twin TWIN bricks away."""

    def __init__(self, **params):
        self.base = tiny_workload(n_frames=4)
        self.intr = self.base.intr
        # blocks of 0.125 m: the shift is a whole number of metres
        self.params = dict(self.base.params, voxel_size=1.0 / 64, mu=1.0 / 16, num_buckets=1 << 10,
                           num_excess=1 << 13, num_blocks=1 << 13, **params)

    def frame(self, k):
        f = self.base.frame(k // 2)
        T = f.T_wc.copy()
        if k & 1:
            T[:3, 3] += TWIN.astype(np.float32)
        return dataclasses.replace(f, T_wc=T)


def _run(itm, w, frames):
    import torch
    g, o = itm.Scene(**w.params), oracle.Scene(**w.params)
    ci = itm.make_intrinsics(w.intr.width, w.intr.height, w.intr.fx, w.intr.fy, w.intr.cx, w.intr.cy)
    V = torch.zeros((w.intr.height, w.intr.width, 4), dtype=torch.float32, device="cuda")
    N = torch.zeros_like(V)
    for k in frames:
        f = w.frame(k)
        g.process(torch.from_numpy(f.depth).cuda(), ci, f.T_wc, V, N)
        o.allocate(f.depth, w.intr.as_array(), f.T_wc)
        o.integrate(f.depth, w.intr.as_array(), f.T_wc)
        vo, no = o.raycast(w.intr.width, w.intr.height, w.intr.as_array(), f.T_wc)
        rep = compare_raycast(V.cpu().numpy(), N.cpu().numpy(), vo, no, f.T_wc)
        assert rep["hits"] > 5000
    assert g.status() == 0
    compare_volumes(g.export(), o.export())
    return g, o, ci, V, N


def test_twin_views_share_every_place(itm):
    """Views and their twins in turn, so that either may own a place."""
    w = Twins()
    g, o, ci, V, N = _run(itm, w, [0, 1, 2, 3, 0, 1, 5, 4])
    c = {tuple(x) for x in g.export(False)[0].tolist()}
    twins = {b for b in c if tuple(np.array(b) + 8 * TWIN) in c}
    assert len(twins) > 300


def test_import_with_shared_places_raycasts_the_same(itm):
    """A volume imported alone and together with its far twin gives the same maps from the same pose."""
    import torch
    w = Twins()
    f = w.frame(0)
    g, _, ci, V, N = _run(itm, w, [0, 2])
    coords, sdf, wgt = g.export()
    g.raycast(ci, f.T_wc, V, N)
    alone = V.clone(), N.clone()
    far = coords.copy()
    far += (8 * TWIN).astype(far.dtype)
    both = itm.Scene(**w.params)
    order = np.random.default_rng(0).permutation(2 * len(coords))
    both.import_blocks(np.concatenate([coords, far])[order], np.concatenate([sdf, sdf[::-1]])[order],
                       np.concatenate([wgt, wgt[::-1]])[order])
    both.raycast(ci, f.T_wc, V, N)
    torch.cuda.synchronize()
    assert torch.equal(V, alone[0]) and torch.equal(N, alone[1])


@pytest.mark.parametrize("idle", [1, 3])
def test_swapping_with_shared_places(itm, idle):
    """Blocks leave and return while their brick's place is the twin's, their own or nobody's."""
    w = Twins()
    g, o, deferred, n_host = run_swapping(itm, w, [0, 1, 0, 1, 3, 2, 0, 5, 4, 1, 0], K=4096, idle=idle,
                                          raycast_every=1)
    c = g.swap_counters()
    assert c["moved_out"] > 500 and c["moved_in"] > 200
