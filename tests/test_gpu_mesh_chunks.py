"""The mesh of blocks with more triangles than a warp lists at a time (256):
voxels of random sign, where a cell has up to five triangles and a block some
1300, against the oracle's mesh (the set of triangles, bit for bit), and with
room for a part of them only."""

import numpy as np
import pytest

import oracle
from synth import tiny_workload
from tests.test_gpu_mesh import canonical, gpu_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weight_mode", [0, 1])
@pytest.mark.parametrize("observed", [1.0, 0.9])
def test_blocks_of_many_triangles(weight_mode, observed):
    import torch
    import paper_1708_00783_gb300 as itm
    rng = np.random.default_rng(5)
    coords = np.stack(np.meshgrid(*[np.arange(-1, 2)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.int16)
    coords = np.concatenate([coords, [[9, 9, 9]]]).astype(np.int16)  # and a block of its own
    sdf = rng.uniform(-1, 1, size=(len(coords), 512)).astype(np.float32)
    wgt = (rng.uniform(size=sdf.shape) < observed).astype(np.float32)
    p = dict(tiny_workload(n_frames=1).params, weight_mode=weight_mode)
    g, o = itm.Scene(**p), oracle.Scene(**p)
    g.import_blocks(coords, sdf, wgt)
    for b, F, W in zip(coords, sdf, wgt):
        o.set_block(b, F, W)
    want = o.mesh()
    assert len(want) > 256 * len(coords) * observed ** 8 * 2  # several lists per block
    got = gpu_mesh(itm, g)
    assert np.array_equal(canonical(got), canonical(want))
    rows = {r.tobytes() for r in canonical(got)}
    for cap in (255, 256, 257, len(want) - 1):
        buf = torch.full((cap + 8, 9), np.nan, device="cuda")
        with pytest.raises(itm.ItmError):
            itm.itm_mesh(g.handle, buf, cap)
        a = buf.cpu().numpy()
        assert np.isnan(a[cap:]).all() and not np.isnan(a[:cap]).any()
        assert all(r.tobytes() in rows for r in canonical(a[:cap]))
