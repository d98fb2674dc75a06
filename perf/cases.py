"""The work that users of this library have it do, as cases that can be timed.

Every case is one pass through the public entry points on a seeded analytic
room (a box of free space with spheres and boxes in it, seen by a moving
pinhole camera with the axial noise and the flying pixels of a structured
light sensor).  Lengths are metres; a pose is camera-to-world, camera +z
forward, +y down.

A live map is in the state: some frames are fused before the call, and the
passes go round a ring of neighbouring frames, as a camera that looks around
in a room it has mapped.
"""

import math

import numpy as np
import torch

import paper_1708_00783_gb300 as itm

DEV = "cuda"


# ------------------------------------------------------------------ the cases

def _frame(name, width, height, voxel_m, u16, **more):
    return dict({"name": name, "kind": "frame", "width": width, "height": height, "voxel_m": voxel_m,
                 "mu_voxels": 4, "u16": u16, "extent_m": 4.0}, **more)


def listed():
    return [
        # The smallest configuration (configs/tiny.json): a robot's or a phone's
        # low-resolution depth stream, where launches and latency count.
        _frame("frame_tiny", 160, 120, 0.010, False),
        # A cropped sensor image: no side is a multiple of a tile.
        _frame("frame_ragged", 333, 247, 0.008, False),
        # The headline: 640x480 millimetre frames at 5 mm (configs/kinect.json).
        _frame("frame_room", 640, 480, 0.005, True),
        # The largest map: a 20 m hall at 2 mm (configs/large.json), hundreds of
        # thousands of visible blocks.
        _frame("frame_hall", 640, 480, 0.002, True, mu_voxels=5, extent_m=20.0),
        # A frame fused with the learned per-pixel weight (weight mode 1).
        dict(_frame("frame_learned", 640, 480, 0.005, False), kind="learned"),
        # A frame of a depth and an RGB camera, and the colour of what is seen.
        dict(_frame("frame_colour", 640, 480, 0.005, True), kind="colour"),
        # A camera turning round with a device array smaller than the map:
        # blocks leave for the host store behind it and return in front.
        dict(_frame("frame_swap", 640, 480, 0.008, True), kind="swap"),
        # The camera pose of a new frame against the last raycast: three pyramid
        # levels, 19 steps (the settings of the benchmark and the tests).
        {"name": "track_room", "kind": "track", "width": 640, "height": 480},
        # The whole map of posed submaps rendered as one.
        {"name": "combined_map", "kind": "combined", "width": 640, "height": 480, "voxel_m": 0.005, "submaps": 6},
        # Many rooms of uneven sizes served in one call.
        {"name": "batch_rooms", "kind": "batch", "scenes": 24},
        # One step of the confidence network's training at its default batch.
        {"name": "train_step", "kind": "train", "samples": 8192},
        # The map exported as a mesh: its size asked for, then the triangles, in
        # an order that does not change from one export to the next.
        {"name": "mesh_room", "kind": "mesh", "width": 640, "height": 480, "voxel_m": 0.005},
    ]


def _between(rng, lo, hi):
    """A whole number, uniform in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "learned", "colour", "swap", "track", "combined", "batch", "train",
                       "mesh"])
    if kind == "batch":
        return {"kind": kind, "scenes": _between(rng, 2, 24)}
    if kind == "train":
        return {"kind": kind, "samples": _between(rng, 200, 8192)}
    width = _between(rng, 96, 640)
    height = max(33, int(width * rng.uniform(0.55, 0.75)))
    case = {"kind": kind, "width": width, "height": height}
    if kind == "track":
        return case
    hall = kind == "frame" and rng.random() < 0.25
    finest = 0.002 if hall else 0.008 if kind == "swap" else 0.0045
    case["voxel_m"] = round(math.exp(rng.uniform(math.log(finest), math.log(0.020))), 4)
    if kind == "combined":
        case["submaps"] = rng.randint(1, 6)
    elif kind != "mesh":
        case.update(mu_voxels=rng.choice([3, 4, 5]), u16=kind != "learned" and rng.random() < 0.5,
                    extent_m=20.0 if hall else 4.0)
    return case


# ------------------------------------------------------- analytic depth frames

def _rng(seed, *more):
    return np.random.default_rng([int(seed) & 0x7fffffff, *more])


class _World:
    """A box of free space with seeded spheres and boxes on its floor and walls."""

    def __init__(self, seed, extent_m):
        r = _rng(seed, 1)
        large = extent_m > 8.0
        size = (extent_m, 3.0 if large else 2.5, extent_m * (0.5 if large else 0.75))
        self.large = large
        self.lo = np.array([-size[0] / 2, 0.0, -size[2] / 2])
        self.hi = np.array([size[0] / 2, size[1], size[2] / 2])
        self.spheres, self.boxes = [], []
        for _ in range(100 if large else 20):
            h = r.uniform(0.05, 0.3)
            c = r.uniform(self.lo + h, self.hi - h)
            axis = r.choice([0, 1, 2], p=[0.3, 0.4, 0.3])
            c[axis] = (self.lo[axis] + h) if axis == 1 or r.random() < 0.5 else (self.hi[axis] - h)
            if r.random() < 0.5:
                self.spheres.append((c, h))
            else:
                e = h * r.uniform(0.6, 1.0, size=3)
                self.boxes.append((c - e, c + e))

    def poses(self, seed, count, yaw_step, move):
        """count poses of a camera that turns by yaw_step and moves by about `move` a frame."""
        r = _rng(seed, 2)
        if self.large:
            p, yaw = np.array([r.uniform(-9.0, -5.0), 1.5, r.uniform(-1.5, 1.5)]), math.pi / 2 + r.uniform(-0.3, 0.3)
        else:
            p, yaw = r.uniform((-1.0, 0.9, -0.6), (1.0, 1.6, 0.6)), r.uniform(0, 2 * math.pi)
        pitch, step = r.uniform(-0.25, 0.0), r.normal(size=3)
        step *= move / np.linalg.norm(step)
        out = []
        for k in range(count):
            a = yaw + yaw_step * k
            f = np.array([math.cos(pitch) * math.sin(a), math.sin(pitch), math.cos(pitch) * math.cos(a)])
            x = np.cross(f, (0.0, 1.0, 0.0))
            x /= np.linalg.norm(x)
            T = np.eye(4)
            T[:3, 0], T[:3, 1], T[:3, 2], T[:3, 3] = x, np.cross(f, x), f, p + step * k
            out.append(T.astype(np.float32))
        return out

    def render(self, cam, poses):
        """Exact z-depth float64 [frames, H, W] on the GPU."""
        dc = _rays(cam)
        T = torch.from_numpy(np.stack(poses).astype(np.float64)).to(DEV)
        D = torch.einsum("hwc,fkc->fhwk", dc, T[:, :3, :3])
        o = T[:, None, None, :3, 3]
        lo, hi = (torch.from_numpy(b).to(DEV) for b in (self.lo, self.hi))
        best = torch.where(D > 0, (hi - o) / D, torch.where(D < 0, (lo - o) / D, math.inf)).amin(-1)
        a = (D * D).sum(-1)
        for c, rad in self.spheres:
            oc = o - torch.from_numpy(c).to(DEV)
            b, q = (D * oc).sum(-1), (oc * oc).sum(-1) - rad * rad
            disc = b * b - a * q
            t = (-b - disc.clamp(min=0).sqrt()) / a
            best = torch.where((disc >= 0) & (t > 0) & (q > 0) & (t < best), t, best)
        for blo, bhi in self.boxes:
            t1, t2 = ((torch.from_numpy(b).to(DEV) - o) / D for b in (blo, bhi))
            tn, tf = torch.minimum(t1, t2).amax(-1), torch.maximum(t1, t2).amin(-1)
            best = torch.where((tn <= tf) & (tn > 0) & (tn < best), tn, best)
        return best


def _camera(width, height):
    """Intrinsics with the field of view of the 640x480 configuration."""
    f = 525.0 * width / 640.0
    return itm.make_intrinsics(width, height, f, f, (width - 1) / 2.0, (height - 1) / 2.0)


def _rays(cam, dtype=torch.float64):
    u = torch.arange(cam.width, device=DEV, dtype=dtype)
    v = torch.arange(cam.height, device=DEV, dtype=dtype)
    x = ((u - cam.cx) / cam.fx)[None, :].expand(cam.height, -1)
    y = ((v - cam.cy) / cam.fy)[:, None].expand(-1, cam.width)
    return torch.stack([x, y, torch.ones_like(x)], -1)


def _sigma(z):
    """Axial noise of a structured-light sensor (Nguyen, Izadi and Lovell, 2012)."""
    return 0.0012 + 0.0019 * (z - 0.4) ** 2


def _measure(z, seed):
    """Millimetre frames as the sensor gives them: noise, flying pixels at depth edges, nothing out of range."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) & 0x7fffffff)
    m = z + _sigma(z) * torch.randn(z.shape, generator=g, device=DEV, dtype=z.dtype)
    right = torch.roll(z, -1, 2)
    pick = ((z - right).abs() > 0.1) & (torch.rand(z.shape, generator=g, device=DEV) < 0.5)
    pick[:, :, -1] = False
    a = torch.rand(z.shape, generator=g, device=DEV, dtype=z.dtype)
    m = torch.where(pick, z + a * (right - z), m)
    m = torch.where((m >= 0.4) & (m <= 5.0), m, 0.0)
    return torch.round(m * 1000.0)


def _to_metres(mm):
    """The float frame of a millimetre frame: the float nearest to mm / 1000."""
    return (mm / 1000.0).to(torch.float32).contiguous()


# ------------------------------------------------------------------- the states

def _tables(voxel_m):
    """Hash and block array sizes: those of the repository's configurations by voxel size."""
    if voxel_m >= 0.008:
        return dict(num_buckets=1 << 17, num_excess=1 << 15, num_blocks=1 << 16)
    if voxel_m >= 0.004:
        return dict(num_buckets=1 << 20, num_excess=1 << 17, num_blocks=1 << 19)
    return dict(num_buckets=1 << 22, num_excess=1 << 18, num_blocks=1 << 21)


def _scene(voxel_m, mu_voxels=4, weight_mode=0, **tables):
    return itm.Scene(voxel_size=voxel_m, mu=mu_voxels * voxel_m, max_w=100, z_min=0.4, z_max=5.0,
                     weight_mode=weight_mode, **(tables or _tables(voxel_m)))


def _maps(cam):
    v = torch.zeros((cam.height, cam.width, 4), dtype=torch.float32, device=DEV)
    return v, torch.zeros_like(v)


BEFORE, RING = 4, 4  # frames fused before the first pass, frames that the passes go round


def _views(case, seed, count=BEFORE + RING, yaw_step=0.06):
    """The camera, the poses and the millimetre frames of a sequence."""
    cam = _camera(case["width"], case["height"])
    world = _World(seed, case.get("extent_m", 4.0))
    poses = world.poses(seed, count, yaw_step, 0.01)
    return cam, poses, _measure(world.render(cam, poses), seed)


def _live(case, seed, ring=RING, before=BEFORE, yaw_step=0.06, weight_mode=0, **tables):
    """A scene, the frames to fuse into it and the ring of frames that the passes go round."""
    cam, poses, mm = _views(case, seed, before + ring, yaw_step)
    scene = _scene(case["voxel_m"], case.get("mu_voxels", 4), weight_mode, **tables)
    depth = [_to_metres(m) for m in mm]
    vertex, normal = _maps(cam)
    s = {"kind": case["kind"], "cam": cam, "scene": scene, "vertex": vertex, "normal": normal, "at": 0,
         "poses": poses[before:], "depth": depth[before:], "u16": bool(case.get("u16"))}
    if s["u16"]:
        s["raw"] = [m.to(torch.int32).to(torch.int16).contiguous() for m in mm[before:]]
        s["float"] = torch.zeros((cam.height, cam.width), dtype=torch.float32, device=DEV)
    s["fuse"] = list(zip(depth[:before], poses[:before]))
    return s


def _init_params(seed):
    """A confidence network's parameters, He-uniform as its training starts (W1, b1, W2, b2, w3, b3)."""
    r, f, h = _rng(seed, 5), itm.ITM_MLP_FEATURES, itm.ITM_MLP_HIDDEN
    parts = [r.uniform(-1, 1, h * f) * math.sqrt(6.0 / f), 0.1 * r.normal(size=h),
             r.uniform(-1, 1, h * h) * math.sqrt(6.0 / h), 0.1 * r.normal(size=h),
             r.uniform(-1, 1, h) * math.sqrt(6.0 / h), r.uniform(-1, 1, 1)]
    return torch.from_numpy(np.concatenate(parts).astype(np.float32)).to(DEV)


def _frame_state(case, seed):
    s = _live(case, seed)
    for d, T in s.pop("fuse"):
        s["scene"].process(d, s["cam"], T)
    return s


def _learned_state(case, seed):
    s = _live(case, seed, weight_mode=1)
    s["packed"] = torch.zeros(itm.ITM_MLP_PACKED_BYTES, dtype=torch.uint8, device=DEV)
    itm.itm_mlp_pack(_init_params(seed), s["packed"])
    s["wpx"] = torch.zeros_like(s["depth"][0])
    for d, T in s.pop("fuse"):
        s["scene"].process_weighted(d, s["packed"], s["wpx"], s["cam"], T)
    return s


def _colour_state(case, seed):
    s = _live(case, seed)
    s["scene"].colour_enable()
    cam = s["cam"]
    # smooth images with sensor noise, from a camera 2 cm beside the depth camera
    g = torch.Generator(device=DEV).manual_seed(int(seed) & 0x7fffffff)
    coarse = torch.rand((len(s["depth"]), 3, 12, 16), generator=g, device=DEV)
    img = 255.0 * torch.nn.functional.interpolate(coarse, size=(cam.height, cam.width), mode="bilinear")
    img = (img + 4.0 * torch.randn(img.shape, generator=g, device=DEV)).clamp(0, 255)
    s["rgb"] = [i.permute(1, 2, 0).to(torch.uint8).contiguous() for i in img]
    s["d2c"] = np.eye(4, dtype=np.float32)
    s["d2c"][0, 3] = 0.02
    s["seen"] = torch.zeros((cam.height, cam.width, 4), dtype=torch.uint8, device=DEV)
    for d, T in s.pop("fuse"):
        s["scene"].allocate(d, cam, T)
        s["scene"].integrate_colour(d, cam, T, s["rgb"][0], cam, s["d2c"])
    return s


def _swap_state(case, seed):
    # a whole turn in 30 frames; the device array holds about half of the room
    # (entry slots for all of it in the host store)
    s = _live(case, seed, ring=30, before=0, yaw_step=2 * math.pi / 30, num_buckets=1 << 16, num_excess=1 << 14,
              num_blocks=1 << 14)
    s.pop("fuse")
    s["scene"].swap_enable(8192, 1)
    for _ in range(len(s["poses"])):
        _run_swap(s)
    return s


def _track_inputs(case, seed):
    """The last view's vertex and normal maps, a new frame from a pose up to 2 cm and 1 degree away."""
    cam = _camera(case["width"], case["height"])
    world = _World(seed, 4.0)
    poses = world.poses(seed, 2, math.radians(_rng(seed, 6).uniform(0.3, 1.0)), 0.02)
    z = world.render(cam, poses)
    depth = _to_metres(_measure(z, seed)[1])
    T = torch.from_numpy(poses[0].astype(np.float64)).to(DEV)
    P = (_rays(cam) * z[0][..., None]) @ T[:3, :3].T + T[:3, 3]
    N = torch.zeros_like(P)
    # along +v times along +u: towards the camera (image y points down)
    N[1:-1, 1:-1] = torch.linalg.cross(P[2:, 1:-1] - P[:-2, 1:-1], P[1:-1, 2:] - P[1:-1, :-2])
    size = N.norm(dim=-1, keepdim=True)
    ok = (size[..., 0] > 0)
    jump = torch.zeros_like(ok)
    jump[1:-1, 1:-1] = ((z[0][2:, 1:-1] - z[0][:-2, 1:-1]).abs() < 0.1) & (
        (z[0][1:-1, 2:] - z[0][1:-1, :-2]).abs() < 0.1)
    ok &= jump
    N = torch.where(ok[..., None], N / size.clamp(min=1e-30), 0.0)
    V4 = torch.cat([P, torch.ones_like(size)], -1).to(torch.float32).contiguous()
    N4 = torch.cat([N, ok[..., None].to(N.dtype)], -1).to(torch.float32).contiguous()
    return cam, depth, V4, N4, poses[0]


TRACK_ITERS, TRACK_THRESH = [10, 5, 4], [0.05, 0.1, 0.2]


def _track_state(case, seed):
    cam, depth, V, N, T_ref = _track_inputs(case, seed)
    size = itm.itm_track_scratch_bytes(cam.width, cam.height, len(TRACK_ITERS))
    scratch = torch.zeros(size + 256, dtype=torch.uint8, device=DEV)
    return {"kind": "track", "cam": cam, "depth": depth, "V": V, "N": N, "T_ref": T_ref, "scratch": scratch,
            "at": scratch.data_ptr() + (-scratch.data_ptr()) % 256}


def _combined_state(case, seed):
    n = case["submaps"]
    cam, poses, mm = _views(case, seed, 3 * n, 0.12)
    r, scenes, P = _rng(seed, 7), [], []
    for i in range(n):
        # submap-from-world: up to 15 degrees about the vertical, up to 0.5 m
        a, M = math.radians(r.uniform(-15, 15)), np.eye(4)
        M[0, 0] = M[2, 2] = math.cos(a)
        M[0, 2], M[2, 0] = math.sin(a), -math.sin(a)
        M[:3, 3] = r.uniform(-0.3, 0.3, size=3)
        sc = _scene(case["voxel_m"])
        for k in range(3 * i, 3 * i + 3):
            sc.process(_to_metres(mm[k]), cam, (M @ poses[k]).astype(np.float32))
        scenes.append(sc)
        P.append(M.astype(np.float32))
    vertex, normal = _maps(cam)
    return {"kind": "combined", "cam": cam, "scenes": scenes, "P": np.stack(P), "T": poses[len(poses) // 2],
            "vertex": vertex, "normal": normal}


_BATCH_SIZES = [(80, 60), (160, 120), (320, 240), (640, 480)]


def _batch_state(case, seed):
    r, rooms = _rng(8), []  # the rooms' sizes are the same for every seed, what is in them is not
    for i in range(case["scenes"]):
        W, H = _BATCH_SIZES[i % len(_BATCH_SIZES)]
        vs = round(float(r.uniform(0.005, 0.020)), 4)
        small = W <= 160
        cam, world = _camera(W, H), _World(seed + 1000 * (i + 1), 4.0)
        poses = world.poses(seed + i, 3, 0.05, 0.01)
        depth = [_to_metres(m) for m in _measure(world.render(cam, poses), seed + i)]
        sc = _scene(vs, 4, num_buckets=1 << (16 if small else 18), num_excess=1 << 15,
                    num_blocks=1 << (15 if small else 17))
        rooms.append((sc, cam, poses, depth, _maps(cam)))
    items = [itm.make_batch_items([(sc.handle, depth[k], cam, poses[k], m[0], m[1])
                                   for sc, cam, poses, depth, m in rooms]) for k in range(3)]
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()  # the frames are there before the other stream reads them
    batch = _Batch(case["scenes"])
    batch.run(items[0], stream)
    return {"kind": "batch", "rooms": rooms, "items": items[1:], "batch": batch, "stream": stream, "at": 0}


class _Batch:
    """Owns an itm_batch handle."""

    def __init__(self, n):
        self.handle = itm.itm_batch_create(n)

    def run(self, items, stream):
        itm.itm_batch_run(self.handle, items, stream)

    def __del__(self):
        itm.itm_batch_destroy(self.handle)


def _train_inputs(case, seed):
    """Features and labels of sampled pixels of one room frame: the 7x7 patch of depth differences and the normal."""
    n, cam = case["samples"], _camera(320, 240)
    world = _World(seed, 4.0)
    z = world.render(cam, world.poses(seed, 1, 0.0, 0.01))
    d = _to_metres(_measure(z, seed))[0]
    ok = torch.nonzero((d > 0).reshape(-1)).reshape(-1)
    g = torch.Generator(device=DEV).manual_seed(int(seed) & 0x7fffffff)
    pix = ok[torch.randint(0, ok.numel(), (n,), generator=g, device=DEV)]
    feat, _ = _features(d, cam, 0.02)
    label = ((d.double() - z[0]).abs() <= 2.0 * _sigma(z[0])).reshape(-1)[pix]
    return feat[pix].to(torch.float32).contiguous(), label.to(torch.float32).contiguous(), _init_params(seed)


def _train_state(case, seed):
    feat, label, params = _train_inputs(case, seed)
    zero = torch.zeros_like(params)
    return {"kind": "train", "feat": feat, "label": label, "params": params, "grad": zero.clone(), "m": zero.clone(),
            "v": zero.clone(), "loss": torch.zeros(1, device=DEV), "step": 0,
            "scratch": torch.zeros(case["samples"] * itm.ITM_MLP_SCRATCH_PER_SAMPLE, device=DEV)}


def _mesh_state(case, seed):
    s = _live(case, seed, ring=1, before=8, yaw_step=0.12)
    for d, T in s.pop("fuse"):
        s["scene"].process(d, s["cam"], T)
    room = int(2000 * _blocks(case))  # several times the triangles of such a map
    s["buffer"] = torch.zeros((room, 9), device=DEV)
    s["sorted"] = torch.zeros((room, 9), device=DEV)
    # odd multipliers that make one 64-bit key of a triangle's nine coordinates
    s["key"] = torch.from_numpy(_rng(9).integers(1 << 40, 1 << 62, size=9) | 1).to(DEV)
    return s


def prepare(case, seed):
    return {"frame": _frame_state, "learned": _learned_state, "colour": _colour_state, "swap": _swap_state,
            "track": _track_state, "combined": _combined_state, "batch": _batch_state, "train": _train_state,
            "mesh": _mesh_state}[case["kind"]](case, seed)


# -------------------------------------------------------------------- the passes

def _next(s):
    k = s["at"]
    s["at"] = (k + 1) % len(s["poses"])
    return k, s["poses"][k]


def _run_frame(s):
    k, T = _next(s)
    if s["u16"]:
        itm.itm_process_frame_u16(s["scene"].handle, s["raw"][k], s["float"], s["cam"], T, s["vertex"], s["normal"])
        return s["vertex"], s["normal"], s["float"]
    s["scene"].process(s["depth"][k], s["cam"], T, s["vertex"], s["normal"])
    return s["vertex"], s["normal"]


def _run_learned(s):
    k, T = _next(s)
    s["scene"].process_weighted(s["depth"][k], s["packed"], s["wpx"], s["cam"], T, s["vertex"], s["normal"])
    return s["vertex"], s["normal"], s["wpx"]


def _allocate(s, k, T):
    if not s["u16"]:
        s["scene"].allocate(s["depth"][k], s["cam"], T)
        return s["depth"][k]
    itm.itm_allocate_u16(s["scene"].handle, s["raw"][k], s["float"], s["cam"], T)
    return s["float"]


def _run_colour(s):
    k, T = _next(s)
    depth = _allocate(s, k, T)
    s["scene"].integrate_colour(depth, s["cam"], T, s["rgb"][k], s["cam"], s["d2c"])
    s["scene"].raycast(s["cam"], T, s["vertex"], s["normal"])
    s["scene"].colour_at(s["vertex"], s["seen"])
    return s["vertex"], s["normal"], s["seen"]


def _run_swap(s):
    k, T = _next(s)
    depth = _allocate(s, k, T)
    s["scene"].swap_in()
    s["scene"].integrate(depth, s["cam"], T)
    s["scene"].raycast(s["cam"], T, s["vertex"], s["normal"])
    s["scene"].swap_out()
    return s["vertex"], s["normal"]


def _run_track(s):
    return itm.itm_track_depth(s["depth"], s["cam"], TRACK_ITERS, TRACK_THRESH, s["V"], s["N"], s["cam"], s["T_ref"],
                               s["T_ref"], s["at"])


def _run_combined(s):
    itm.itm_raycast_combined([sc.handle for sc in s["scenes"]], s["P"], s["cam"], s["T"], s["vertex"], s["normal"])
    return s["vertex"], s["normal"]


def _run_batch(s):
    k = s["at"]
    s["at"] = (k + 1) % len(s["items"])
    s["batch"].run(s["items"][k], s["stream"])
    return [m for room in s["rooms"] for m in room[4]]


def _run_train(s):
    n = s["label"].numel()
    itm.itm_mlp_loss_grad(s["params"], s["feat"], s["label"], n, s["scratch"], s["grad"], s["loss"])
    s["step"] += 1
    itm.itm_mlp_adam(s["params"], s["grad"], s["m"], s["v"], s["step"], 3e-3)
    return {k: s[k] for k in ("loss", "grad", "params", "m", "v")}


def _run_mesh(s):
    n = itm.itm_mesh(s["scene"].handle)
    if n > s["buffer"].shape[0]:
        s["buffer"], s["sorted"] = (torch.zeros((n, 9), device=DEV) for _ in range(2))
    itm.itm_mesh(s["scene"].handle, s["buffer"], s["buffer"].shape[0])
    tri = s["buffer"][:n]
    order = torch.argsort((tri.view(torch.int32) * s["key"]).sum(1))
    torch.index_select(tri, 0, order, out=s["sorted"][:n])
    return n, s["sorted"]


def run(state):
    return {"frame": _run_frame, "learned": _run_learned, "colour": _run_colour, "swap": _run_swap,
            "track": _run_track, "combined": _run_combined, "batch": _run_batch, "train": _run_train,
            "mesh": _run_mesh}[state["kind"]](state)


# ---------------------------------------------------------------------- the work

def _blocks(case):
    """About how many blocks a view of the room touches: the surface seen (at about 1.6 m, 3.6 m in a hall) in block
    faces, as deep as the truncation band and the noise reach."""
    z = 3.6 if case.get("extent_m", 4.0) > 8.0 else 1.6
    f, block = 525.0 * case["width"] / 640.0, 8 * case["voxel_m"]
    depth = 1.0 + 2 * case.get("mu_voxels", 4) / 8 + 2 * _sigma(z) / block
    return depth * case["width"] * case["height"] * (z / f) ** 2 / block ** 2


def work(case):
    kind = case["kind"]
    if kind == "train":
        # forward and backward: three products of each layer's weights with the samples; parameters and moments
        n = case["samples"]
        return {"bytes": n * 53 * 4 + 7 * 7617 * 4, "flops": 6.0 * n * (52 * 64 + 64 * 64 + 64)}
    if kind == "batch":
        per = [work({"kind": "frame", "width": w, "height": h, "voxel_m": 0.0125, "u16": False})
               for w, h in _BATCH_SIZES]
        return {k: case["scenes"] * sum(p[k] for p in per) / len(per) for k in ("bytes", "flops")}
    px = case["width"] * case["height"]
    if kind == "track":
        # the depth frame and the reference maps once; 19 steps over three levels at about 200 operations a pixel
        return {"bytes": px * 36, "flops": px * 200.0 * (10 + 5 / 4 + 4 / 16)}
    if kind == "combined":
        # the voxels around the surface (two layers of each visible block, sdf and weight) of each submap, the maps
        return {"bytes": px * 32 + _blocks(case) * case["submaps"] * 128 * 5, "flops": px * 2000.0 * case["submaps"]}
    if kind == "mesh":
        # every block's voxels once, about 100 triangles a block
        blocks = 3 * _blocks(case)
        return {"bytes": blocks * (512 * 5 + 100 * 36), "flops": blocks * 512 * 20.0}
    # a frame: the depth in, the maps out, ten bytes for each of about 300 updated voxels a block
    per_voxel = {"frame": 10, "learned": 16, "colour": 14, "swap": 10}[kind]
    per_pixel = 32 + (6 if case["u16"] else 4) + {"frame": 0, "learned": 4, "colour": 23, "swap": 0}[kind]
    flops = px * 2000.0 + _blocks(case) * 300 * 60.0
    if kind == "learned":
        flops += px * 2.0 * (52 * 64 + 64 * 64 + 64)
    return {"bytes": px * per_pixel + _blocks(case) * 300 * per_voxel, "flops": flops}


# ------------------------------------------------------------- in 64 bits

def _features(d, cam, mu):
    """The 52 features of every pixel of a depth frame (float64 [pixels, 52]) and the pixels that have depth."""
    D = torch.where(d > 0, d, 0.0).double()
    patch = torch.nn.functional.unfold(D[None, None], 7, padding=3)[0].T  # pixels x 49, row by row
    x = torch.where(patch > 0, ((patch - D.reshape(-1, 1)) / mu).clamp(-4, 4), 0.0)
    P = _rays(cam) * D[..., None]
    a, b = torch.zeros_like(P), torch.zeros_like(P)
    a[1:-1], b[:, 1:-1] = P[2:] - P[:-2], P[:, 2:] - P[:, :-2]
    n = torch.linalg.cross(a, b)
    has = torch.zeros_like(D, dtype=torch.bool)
    has[1:-1, 1:-1] = (D[2:, 1:-1] > 0) & (D[:-2, 1:-1] > 0) & (D[1:-1, 2:] > 0) & (D[1:-1, :-2] > 0)
    size = n.norm(dim=-1, keepdim=True)
    n = torch.where(has[..., None] & (size > 0), n / size.clamp(min=1e-300), 0.0)
    ok = (D > 0).reshape(-1, 1)
    return torch.where(ok, torch.cat([x, n.reshape(-1, 3)], 1), 0.0), ok[:, 0]


def _bf16(x):
    """The network's weights and the inputs of its products are bfloat16 values."""
    return x.to(torch.float32).to(torch.bfloat16).double()


def _split(p):
    f, h = itm.ITM_MLP_FEATURES, itm.ITM_MLP_HIDDEN
    W1, b1, W2, b2, w3, b3 = torch.split(p.double(), [h * f, h, h * h, h, h, 1])
    return _bf16(W1).reshape(h, f), b1, _bf16(W2).reshape(h, h), b2, w3, b3


def _forward(p, feat):
    W1, b1, W2, b2, w3, b3 = _split(p)
    h1 = _bf16((_bf16(feat) @ W1.T + b1).clamp(min=0))
    h2 = (h1 @ W2.T + b2).clamp(min=0)
    return h1, h2, h2 @ w3 + b3


def _exact_train(case, seed):
    feat, y, p = _train_inputs(case, seed)
    n, y = y.numel(), y.double()
    W1, _, W2, _, w3, _ = _split(p)
    h1, h2, o = _forward(p, feat)
    loss = (torch.nn.functional.softplus(o) - o * y).mean()
    do = (torch.sigmoid(o) - y) / n
    d2 = torch.where(h2 > 0, do[:, None] * w3, 0.0)
    d1 = torch.where(h1 > 0, d2 @ W2, 0.0)
    grad = torch.cat([(d1.T @ _bf16(feat)).reshape(-1), d1.sum(0), (d2.T @ h1).reshape(-1), d2.sum(0), do @ h2,
                      do.sum()[None]])
    # the first step of Adam (0.9, 0.999, 1e-8) from zero moments
    m, v = 0.1 * grad, 0.001 * grad * grad
    return {"loss": loss[None], "grad": grad, "params": p.double() - 3e-3 * grad / (grad.abs() + 1e-8), "m": m, "v": v}


def _exact_learned(case, seed):
    cam, _, mm = _views(case, seed)
    feat, ok = _features(_to_metres(mm[BEFORE]), cam, case["mu_voxels"] * case["voxel_m"])
    w = torch.where(ok, torch.sigmoid(_forward(_init_params(seed), feat)[2]), 0.0)
    return None, None, w.reshape(cam.height, cam.width)


def _exact_track(case, seed):
    """Point-to-plane alignment by Gauss-Newton, coarse to fine, every operation in 64 bits."""
    cam, depth, V4, N4, T_ref = _track_inputs(case, seed)
    levels = [(depth.double(), cam.fx, cam.fy, cam.cx, cam.cy)]
    for _ in TRACK_ITERS[1:]:
        d, fx, fy, cx, cy = levels[-1]
        h, w = d.shape[0] // 2, d.shape[1] // 2
        q = d[:2 * h, :2 * w].reshape(h, 2, w, 2).permute(0, 2, 1, 3).reshape(h, w, 4)
        n = (q > 0).sum(-1)
        levels.append((torch.where(n > 0, q.clamp(min=0).sum(-1) / n.clamp(min=1), 0.0), fx / 2, fy / 2,
                       (cx - 0.5) / 2, (cy - 0.5) / 2))
    V, N = V4.double().reshape(-1, 4), N4.double().reshape(-1, 4)
    T = torch.from_numpy(np.asarray(T_ref, np.float64)).to(DEV)
    R0, t0 = T[:3, :3].clone(), T[:3, 3].clone()
    steps = 0
    for l in reversed(range(len(levels))):
        d, fx, fy, cx, cy = levels[l]
        v, u = torch.meshgrid(torch.arange(d.shape[0], device=DEV), torch.arange(d.shape[1], device=DEV),
                              indexing="ij")
        pc = torch.stack([(u - cx) / fx * d, (v - cy) / fy * d, d], -1)[d > 0]
        for _ in range(TRACK_ITERS[l]):
            pw = pc @ T[:3, :3].T + T[:3, 3]
            pr = (pw - t0) @ R0
            ur, vr = cam.fx * pr[:, 0] / pr[:, 2] + cam.cx, cam.fy * pr[:, 1] / pr[:, 2] + cam.cy
            ok = (pr[:, 2] > 0) & (ur >= 0) & (ur <= cam.width - 1) & (vr >= 0) & (vr <= cam.height - 1)
            at = torch.where(ok, (vr + 0.5).long() * cam.width + (ur + 0.5).long(), 0)
            Vp, Np = V[at], N[at]
            e = pw - Vp[:, :3]
            ok &= (Vp[:, 3] > 0) & (Np[:, 3] > 0) & ((e * e).sum(-1) <= TRACK_THRESH[l] ** 2)
            n = Np[:, :3]
            J = torch.where(ok[:, None], torch.cat([torch.linalg.cross(pw, n), n], -1), 0.0)
            r = torch.where(ok, (e * n).sum(-1), 0.0)
            x = torch.linalg.solve(J.T @ J, -(J.T @ r))
            K = torch.zeros((4, 4), dtype=torch.float64, device=DEV)
            K[0, 1], K[0, 2], K[1, 2] = -x[2], x[1], -x[0]
            K[1, 0], K[2, 0], K[2, 1] = x[2], -x[1], x[0]
            S = torch.linalg.matrix_exp(K)
            S[:3, 3] = x[3:]
            T = S @ T
            steps += 1
    return T, steps


def exact(case, seed):
    """The outputs that are sums and products of the inputs.  The vertex and normal maps, and the mesh of a fused map,
    are what the method's single-precision arithmetic decides step by step (which voxel is updated, where a ray
    steps): 64 bits would be another computation, and they have no value here."""
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "learned":
        return _exact_learned(case, seed)
    if case["kind"] == "track":
        return _exact_track(case, seed)
    if case["kind"] == "frame" and case["u16"]:
        return None, None, _views(case, seed)[2][BEFORE] / 1000.0
    return None
