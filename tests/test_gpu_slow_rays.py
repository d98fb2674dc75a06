"""Raycasts with rays that are not through after the first phase's iterations.

With a band of one voxel the fine search takes many steps, and from a pose that
the map was not built from, rays skim walls and cross gaps: both go through the
slow list, where four lanes march one ray.  The maps are compared with the
oracle (the bars of parity_util.py), and with the batch, which marches every
ray in its tile: those are equal bit for bit.  Sizes: a part of a tile, a few
ragged tiles, more slow rays than the second phase takes at once, and a strip.
Each map is taken twice, as the counts of a raycast are kept in two sets."""

import numpy as np
import pytest

import oracle
from synth import Intrinsics, tiny_workload
from tests.parity_util import compare_raycast

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("band_voxels", [1, 4])
@pytest.mark.parametrize("size", [(5, 3), (33, 21), (160, 120), (1024, 20), (1280, 960)])
def test_slow_rays(size, band_voxels):
    import torch
    import paper_1708_00783_gb300 as itm
    w = tiny_workload(n_frames=10)
    i = w.intr
    wi = itm.make_intrinsics(i.width, i.height, i.fx, i.fy, i.cx, i.cy)
    W, H = size
    sx = max(W / i.width, H / i.height) if W * H > 1000 else 1.0  # small images are crops of the view
    c = Intrinsics(W, H, i.fx * sx, i.fy * sx, W / 2.0 - 0.5, H / 2.0 - 0.5)
    ci = itm.make_intrinsics(W, H, c.fx, c.fy, c.cx, c.cy)
    p = dict(w.params, mu=band_voxels * w.params["voxel_size"])
    g, b, o = itm.Scene(**p), itm.Scene(**p), oracle.Scene(**p)
    batch = itm.itm_batch_create(1)
    stream = torch.cuda.Stream()
    for k in range(2):
        f = w.frame(k)
        D = torch.from_numpy(f.depth).cuda()
        for s in (g, b):
            s.allocate(D, wi, f.T_wc)
            s.integrate(D, wi, f.T_wc)
        o.process(f.depth, i.as_array(), f.T_wc, raycast=False)
    nothing = torch.zeros((H, W), device="cuda")  # a frame without depth leaves the map as it is
    for k in (0, 5, 9):
        T = w.frame(k).T_wc
        maps = [torch.full((H, W, 4), 7.0, device="cuda") for _ in range(6)]
        for m in range(2):
            g.raycast(ci, T, maps[2 * m], maps[2 * m + 1])
        torch.cuda.synchronize()
        itm.itm_batch_run(batch, itm.make_batch_items([(b.handle, nothing, ci, T, maps[4], maps[5])]), stream)
        stream.synchronize()
        for m in (0, 1):
            assert torch.equal(maps[m], maps[2 + m]) and torch.equal(maps[m], maps[4 + m]), (k, m)
        vo, no = o.raycast(W, H, c.as_array(), T)
        v, n = maps[0].cpu().numpy(), maps[1].cpu().numpy()
        if v.size > 4000:
            compare_raycast(v, n, vo, no, T)
        else:  # fewer pixels than the bar's share has room for: all equal
            assert np.array_equal(v[..., 3], vo[..., 3]) and np.abs(v - vo).max() < 1e-4
    itm.itm_batch_destroy(batch)
