"""The tracker's step kernel at its edges: image sizes around one CTA, around
one pixel per thread of every CTA and around its four-pixel passes, and the
warp-wide solve against the host's step.

Sums: the bound of test_gpu_track.py (2e-6 of the magnitude of the terms; a
thread adds at most four to eight products here).  Solve: both sides work in
double on the same sums, so the poses differ by the float rounding of their
elements (|T| < 8: half an ulp each, 2 x 2^-22) plus the double solves' error,
cond(H) 2^-52 relative, below that for the systems here."""

import numpy as np
import pytest

import oracle
from synth import Intrinsics
from tests.test_oracle_track_pins import exp_pose

pytestmark = pytest.mark.gpu


def _case(W, H, seed=0):
    """A curved surface z(x, y) seen from the reference, and its maps."""
    intr = Intrinsics(W, H, 0.8 * W, 0.8 * W, (W - 1) / 2, (H - 1) / 2)
    u, v = np.meshgrid(np.arange(W), np.arange(H))
    x, y = (u - intr.cx) / intr.fx, (v - intr.cy) / intr.fy
    z = 2.0 + 0.3 * np.sin(3 * x) * np.cos(2 * y) + 0.2 * x * y
    P = np.stack([x * z, y * z, z], -1)
    du, dv = np.gradient(P, axis=1), np.gradient(P, axis=0)
    n = np.cross(dv, du)
    n /= np.linalg.norm(n, axis=-1, keepdims=True)
    one = np.ones((H, W, 1))
    V = np.concatenate([P, one], -1).astype(np.float32)
    N = np.concatenate([n, one], -1).astype(np.float32)
    rng = np.random.default_rng(seed)
    d = z.astype(np.float32)
    d[rng.uniform(size=d.shape) < 0.05] = 0.0
    return intr, d, V, N


@pytest.mark.parametrize("W,H", [(3, 3), (16, 32), (19, 27), (311, 251), (640, 487), (1024, 640)])
def test_sums_at_grid_edges(W, H):
    import torch
    import paper_1708_00783_gb300 as itm
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


@pytest.mark.parametrize("W,H,angle", [(40, 30, 0.01), (320, 240, 0.05), (320, 240, 0.6), (640, 480, 0.002)])
def test_device_step_is_the_host_step(W, H, angle):
    """One step from a pose `angle` off (0.6 rad: the sine and cosine themselves, not their series)."""
    import torch
    import paper_1708_00783_gb300 as itm
    intr, d, V, N = _case(W, H, 1)
    ci = itm.make_intrinsics(W, H, intr.fx, intr.fy, intr.cx, intr.cy)
    dev = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    dd, Vd, Nd = dev(d), dev(V), dev(N)
    Tref = np.eye(4, dtype=np.float32)
    Tg = exp_pose(np.array([0.0, 0.0, angle, 0.02, -0.01, 0.01]), Tref).astype(np.float32)
    work = torch.zeros(itm.ITM_ICP_WORK_DOUBLES, dtype=torch.float64, device="cuda")
    itm.itm_icp_reduce(dd, ci, Tg, Vd, Nd, ci, Tref, 1.0, work)
    torch.cuda.synchronize()
    Th, x = itm.itm_icp_step(work[:29].cpu().numpy(), Tg)
    nbytes = itm.itm_track_scratch_bytes(W, H, 1)
    scratch = torch.empty(nbytes + 256, dtype=torch.uint8, device="cuda")
    Td, steps = itm.itm_track_depth(dd, ci, [1], [1.0], Vd, Nd, ci, Tref, Tg,
                                    scratch.data_ptr() + (-scratch.data_ptr()) % 256)
    assert steps == 1 and np.abs(Th).max() < 8.0
    if angle > 0.5:
        assert np.linalg.norm(x[:3]) > 0.25
    assert np.abs(Td - Th).max() <= 2.0 ** -21, np.abs(Td - Th).max()
