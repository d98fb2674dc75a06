"""Allocation along segments of one to many blocks, against the oracle.

The enumeration looks up four blocks of a pixel's segment at a time, so the
bands here are a part of a block, about a block (the usual one) and many blocks
deep, on images whose sides are no multiple of a tile; with few buckets most
requests lose theirs and go through the overflow list.  The counts of an
allocation are kept in two sets that take turns: frames are allocated several
times in a row, a repeated frame requests nothing, and a batch in between uses
the same sets."""

import numpy as np
import pytest

import oracle
from synth import Intrinsics, tiny_workload
from tests.parity_util import compare_volumes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("band_voxels", [1, 4, 24, 60])
@pytest.mark.parametrize("size,buckets", [((33, 21), 1 << 16), ((160, 120), 1 << 16), ((97, 50), 1 << 6)])
def test_blocks_of_a_segment(band_voxels, size, buckets):
    import torch
    import paper_1708_00783_gb300 as itm
    w = tiny_workload(n_frames=4)
    W, H = size
    u0, v0 = (w.intr.width - W) // 2, (w.intr.height - H) // 2
    c = Intrinsics(W, H, w.intr.fx, w.intr.fy, w.intr.cx - u0, w.intr.cy - v0)
    ci = itm.make_intrinsics(W, H, c.fx, c.fy, c.cx, c.cy)
    p = dict(w.params, mu=band_voxels * w.params["voxel_size"], num_buckets=buckets, num_excess=1 << 16)
    g, o = itm.Scene(**p), oracle.Scene(**p)
    batch = itm.itm_batch_create(1)
    stream = torch.cuda.Stream()
    for k in range(4):
        f = w.frame(k)
        d = np.ascontiguousarray(f.depth[v0:v0 + H, u0:u0 + W])
        D = torch.from_numpy(d).cuda()
        before = g.stats()["allocated_blocks"]
        if k == 2:
            torch.cuda.synchronize()
            itm.itm_batch_run(batch, itm.make_batch_items([(g.handle, D, ci, f.T_wc, None, None)]), stream)
            stream.synchronize()
        else:
            g.allocate(D, ci, f.T_wc)
        s = g.stats()
        new = s["allocated_blocks"] - before
        assert s["last_requests"] <= new <= s["last_requests"] + s["last_overflow"]
        if k != 2:
            g.allocate(D, ci, f.T_wc)
            again = g.stats()
            assert again["last_requests"] == again["last_overflow"] == 0
            assert again["allocated_blocks"] == s["allocated_blocks"]
            g.integrate(D, ci, f.T_wc)
        o.allocate(d, c.as_array(), f.T_wc)
        o.integrate(d, c.as_array(), f.T_wc)
        assert g.status() == 0 and o.status == 0
        compare_volumes(g.export(), o.export())
    itm.itm_batch_destroy(batch)
