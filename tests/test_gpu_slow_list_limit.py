"""The raycast around the size of its slow list (2^21 pixels): an image of as
many pixels, whose slow rays all find room, and larger ones, whose rays are
marched to their end in their tiles. Both against the batch, which marches
every ray in its tile (and is compared with the oracle at smaller sizes in
test_gpu_slow_rays.py): the arithmetic is the same, so the maps are equal bit
for bit. Each map is taken twice, as the counts are kept in two sets."""

import pytest

from synth import Intrinsics, tiny_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("band_voxels", [1, 4])
@pytest.mark.parametrize("size", [(2048, 1024), (2049, 1024), (1531, 1373)])
def test_around_the_limit(size, band_voxels):
    import torch
    import paper_1708_00783_gb300 as itm
    w = tiny_workload(n_frames=10)
    i = w.intr
    wi = itm.make_intrinsics(i.width, i.height, i.fx, i.fy, i.cx, i.cy)
    W, H = size
    s = max(W / i.width, H / i.height)
    c = Intrinsics(W, H, i.fx * s, i.fy * s, W / 2.0 - 0.5, H / 2.0 - 0.5)
    ci = itm.make_intrinsics(W, H, c.fx, c.fy, c.cx, c.cy)
    p = dict(w.params, mu=band_voxels * w.params["voxel_size"])
    g, b = itm.Scene(**p), itm.Scene(**p)
    batch = itm.itm_batch_create(1)
    for k in range(2):
        f = w.frame(k)
        D = torch.from_numpy(f.depth).cuda()
        for x in (g, b):
            x.allocate(D, wi, f.T_wc)
            x.integrate(D, wi, f.T_wc)
    nothing = torch.zeros((H, W), device="cuda")  # a frame without depth leaves the map as it is
    for k in (0, 9):
        T = w.frame(k).T_wc
        maps = [torch.full((H, W, 4), 7.0, device="cuda") for _ in range(6)]
        for m in range(2):
            g.raycast(ci, T, maps[2 * m], maps[2 * m + 1])
        itm.itm_batch_run(batch, [(b.handle, nothing, ci, T, maps[4], maps[5])])
        torch.cuda.synchronize()
        assert int((maps[0][..., 3] > 0).sum()) > W * H // 20
        for m in (0, 1):
            assert torch.equal(maps[m], maps[2 + m]) and torch.equal(maps[m], maps[4 + m]), (k, m)
    assert g.status() == 0
    itm.itm_batch_destroy(batch)
