"""What a user of this framework has it do, as measurable cases.

A case is one call (or the few calls that belong together) of the package's public entry points on a
map that is already in use: some scans of the same drive have been integrated before, so the voxels
hold values and weights. Scenes, sensors, windows and truncation distances are those of the package's
synthetic workloads (box room, outdoor drive with an OS1-128-shaped sensor, high-resolution corridor,
uneven batches, served sessions); the range noise and the poses come from the seed. The scans are cast
against the scene's analytic primitives on the GPU, which makes them quick to produce.

listed() gives the fixed cases, draw() more of the same ranges, prepare() what a program holds before
the call, run() one pass, work() what a pass cannot do without, exact() the result in 64 bits where the
outputs are computed numbers (voxel grids and counters are whole numbers).
"""
import math

import numpy as np
import torch

from paper_2310_05766_gb300 import binding as b
from paper_2310_05766_gb300 import synth

SIGMA = 0.01            # range noise of the synthetic sensors, metres
REGISTER_STEPS = 6      # Gauss-Newton steps of a registration call


# ---------------------------------------------------------------- cases

def _case(name, kind, scene, beams, azimuths, dims, voxel, tau, **more):
    c = dict(kind=kind, scene=scene, beams=beams, azimuths=azimuths, dx=dims[0], dy=dims[1], dz=dims[2],
             voxel=voxel, tau=tau, reduce=0, flags=0, count=1, step=0)
    c.update(more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a 16-line scanner in a room; launches and latency are what a user waits for
        _case("room_16x360", "integrate", "room", 16, 360, (256, 256, 64), 0.05, 0.2),
        # a robot's loop that may not allocate: fixed memory, a small window, the paper's literal reading
        # (smallest distance of all rays, a step's own distance), invalid returns already dropped by the
        # driver, so the number of points is whatever is left
        _case("static_32x900_min_step", "static", "outdoor", 32, 900, (128, 128, 128), 0.1, 0.4, reduce=1, flags=1),
        # the ordinary call: one scan of an OS1-128-shaped sensor, points on the device
        _case("outdoor_128x1024", "integrate", "outdoor", 128, 1024, (512, 512, 128), 0.064, 0.6),
        # the largest window and scan of the repository: 2 cm voxels, 262 k points
        _case("corridor_128x2048", "integrate", "corridor", 128, 2048, (1024, 1024, 256), 0.02, 0.1),
        # the same ordinary scan end to end: points in pinned host memory, counters read after the scan
        _case("host_128x1024", "host", "outdoor", 128, 1024, (512, 512, 128), 0.064, 0.6),
        # several large maps on one device: the sparse per-scan accumulator
        _case("pool_64x1024", "pool", "outdoor", 64, 1024, (512, 512, 128), 0.064, 0.6),
        # many maps advanced together by one launch, scans and windows of uneven size
        _case("batch_32_maps", "batch", "outdoor", 0, 0, (512, 512, 128), 0.064, 0.6, count=32),
        # a burst of served sessions: 16 requests queued at once from pinned memory, all waited for
        _case("serve_16_sessions", "serve", "outdoor", 0, 0, (512, 512, 128), 0.064, 0.6, count=16),
        # a drive: the window moves a metre, a scan is integrated, and back over ground already mapped
        _case("drive_1m_and_back", "drive", "outdoor", 128, 1024, (512, 512, 128), 0.064, 0.6, step=16),
        # consumers of the map: triangles of its surface,
        _case("mesh_outdoor", "mesh", "outdoor", 128, 1024, (512, 512, 128), 0.064, 0.6),
        # its zero crossings as points,
        _case("surface_outdoor", "surface", "outdoor", 128, 1024, (512, 512, 128), 0.064, 0.6),
        # and a scan registered against it
        _case("register_128x1024", "register", "outdoor", 128, 1024, (512, 512, 128), 0.064, 0.6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["integrate", "integrate", "integrate", "static", "host", "pool", "batch", "serve", "drive", "mesh",
                       "surface", "register"])
    # paper's default reading most of the time, its alternatives otherwise
    reduce, flags = rng.choice([(0, 0), (0, 0), (1, 0), (1, 1), (0, 2), (0, 1)])
    if kind in ("batch", "serve"):
        return _case(None, kind, "outdoor", 0, 0, (512, 512, 128), rng.choice([0.05, 0.064, 0.08, 0.1]),
                     round(rng.uniform(0.2, 0.6), 3), reduce=reduce, flags=flags, count=_log_int(rng, 2, 24))
    scene = rng.choice(["room", "outdoor", "outdoor", "corridor"])
    beams, azimuths = _log_int(rng, 8, 128), _log_int(rng, 180, 2048)
    tau = round(rng.uniform(0.2, 0.6), 3)
    if kind == "register":
        return _case(None, kind, "outdoor", beams, azimuths, (512, 512, 128), 0.064, max(tau, 0.3))
    if kind == "static":
        dims, voxel = rng.choice([((128, 128, 128), 0.1), ((256, 256, 32), 0.08), ((64, 128, 64), 0.2)])
        return _case(None, kind, scene, beams, min(azimuths, 1024), dims, voxel, max(tau, 2 * voxel), reduce=reduce,
                     flags=flags)
    if scene == "corridor" and kind in ("integrate", "host", "pool"):
        return _case(None, kind, scene, beams, azimuths, (1024, 1024, 256), 0.02, round(rng.uniform(0.06, 0.15), 3),
                     reduce=reduce, flags=flags)
    dims = rng.choice([(256, 256, 64), (256, 256, 256), (512, 512, 128), (512, 256, 64)])
    voxel = rng.choice([0.05, 0.064, 0.08, 0.1] if dims[2] > 64 else [0.08, 0.1])   # (the ground lies in the window)
    return _case(None, kind, scene, beams, azimuths, dims, voxel, max(tau, 2 * voxel), reduce=reduce, flags=flags,
                 step=8 * rng.randint(1, 4) if kind == "drive" else 0)


# ---------------------------------------------------------------- inputs

_VFOV = {"room": 30.0, "outdoor": 45.0, "corridor": 45.0}
_RANGE = {"room": (0.3, 20.0), "outdoor": (0.5, 100.0), "corridor": (0.5, 100.0)}


def _cuda64(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _cast(scene, origin, d):
    """Distance along unit directions d (n, 3) from `origin` to the scene's first surface (inf: none)."""
    o = _cuda64(origin)
    inf = torch.full((d.shape[0],), math.inf, dtype=torch.float64, device="cuda")
    best = inf
    inv = 1.0 / d
    if scene.room is not None:      # the walls of a hollow box, seen from inside
        t1, t2 = (_cuda64(scene.room[:3]) - o) * inv, (_cuda64(scene.room[3:]) - o) * inv
        best = torch.minimum(best, torch.maximum(t1, t2).amin(1))
    if scene.ground_z is not None:
        s = (scene.ground_z - o[2]) * inv[:, 2]
        best = torch.minimum(best, torch.where((d[:, 2] < 0) & (s > 0), s, inf))
    for part in _cuda64(scene.boxes).split(16) if len(scene.boxes) else ():
        t1, t2 = (part[:, :3] - o) * inv[:, None], (part[:, 3:] - o) * inv[:, None]
        near, far = torch.minimum(t1, t2).amax(2), torch.maximum(t1, t2).amin(2)
        best = torch.minimum(best, torch.where((far >= near) & (near > 0), near, inf[:, None]).amin(1))
    for part in _cuda64(scene.cylinders).split(16) if len(scene.cylinders) else ():   # upright posts: their sides
        ox, oy = o[0] - part[:, 0], o[1] - part[:, 1]
        a = (d[:, :1] ** 2 + d[:, 1:2] ** 2).clamp_min(1e-300)
        h = d[:, :1] * ox + d[:, 1:2] * oy
        disc = h * h - a * (ox * ox + oy * oy - part[:, 2] ** 2)
        s = (-h - disc.clamp_min(0).sqrt()) / a
        z = o[2] + s * d[:, 2:]
        hit = (disc >= 0) & (s > 0) & (z >= part[:, 3]) & (z <= part[:, 4])
        best = torch.minimum(best, torch.where(hit, s, inf[:, None]).amin(1))
    return best


def _scan(case, scene, R, t, gen, dense=False):
    """One scan from pose (R, t): float32 (n, 4) points in the sensor frame on the GPU, NaN where a beam
    has no return (dense: those dropped)."""
    half = 0.5 * _VFOV[case["scene"]]
    d = _cuda64(synth.beam_directions(case["beams"], case["azimuths"], -half, half))
    Rt = _cuda64(R)
    dw = d[:, :1] * Rt[:, 0] + d[:, 1:2] * Rt[:, 1] + d[:, 2:] * Rt[:, 2]
    rho = _cast(scene, t, dw)
    noise = torch.randn(d.shape[0], dtype=torch.float64, device="cuda", generator=gen).clamp(-3, 3) * SIGMA
    hit = rho <= _RANGE[case["scene"]][1]
    pts = torch.zeros((d.shape[0], 4), dtype=torch.float32, device="cuda")
    pts[:, :3] = torch.where(hit[:, None], d * (rho + noise)[:, None], torch.full_like(d, math.nan)).float()
    return pts[hit].contiguous() if dense else pts


def _scene_and_poses(case, seed, n):
    rng = synth.SplitMix64(seed * 1000003 + 17)
    if case["scene"] == "room":
        yaw, dx, dy = (float(rng.uniform(1, -1.0, 1.0)[0]) for _ in range(3))
        poses = [(synth.rot_zyx(math.pi * yaw + 0.02 * i), np.array([0.6 * dx + 0.02 * i, 0.6 * dy, 0.0])) for i in range(n)]
        return synth.box_room_scene(), poses
    if case["scene"] == "corridor":
        poses = synth.trajectory(n, 0.5, 0.1, seed + 1, wobble_deg=0.3, lateral=0.2, straight_x=True)
        return synth.corridor_scene(seed + 1), poses
    poses = synth.trajectory(n, 1.0, 0.1, seed + 1)
    return synth.outdoor_scene(seed + 1, np.array([t[:2] for _, t in poses])), poses


def _params(case, centre):
    dims = (case["dx"], case["dy"], case["dz"])
    rmin, rmax = _RANGE[case["scene"]]
    return synth.params_dict(dims, case["voxel"], case["tau"], 64, synth.delta_z_for(_VFOV[case["scene"]], case["beams"]),
                             rmin, rmax, case["reduce"], synth.window_origin(centre, dims, case["voxel"]), case["flags"])


class _DeviceWords:
    """A map's voxel grid as the library exposes it: 32-bit words in device memory. `owner` is the object
    that frees the map; a tensor made from this keeps it alive."""

    def __init__(self, handle, params, owner):
        self.owner = owner
        n = int(np.prod(params["dims"], dtype=np.int64))
        self.__cuda_array_interface__ = dict(shape=(n,), typestr="<i4", data=(b.tsdf_grid_device_ptr(handle), False),
                                             version=3, strides=None)


def _grid(handle, params, owner):
    return torch.as_tensor(_DeviceWords(handle, params, owner), device="cuda")


def _map_in_use(case, seed, scans=3, dense=False):
    """A map with the drive's earlier scans integrated, its parameters, and the next scan with its pose."""
    scene, poses = _scene_and_poses(case, seed, scans)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    params = _params(case, poses[-1][1])
    pts = [_scan(case, scene, R, t, gen, dense) for R, t in poses]
    p12 = [synth.pose12(R, t) for R, t in poses]
    m = None
    if case["kind"] != "static":
        m = b.TsdfMap(params)
        if case["kind"] == "pool":
            b.tsdf_set_option(m.handle, b.TSDF_OPT_REDUCTION, b.TSDF_REDUCTION_POOL)
        for p, q in zip(pts[:-1], p12[:-1]):
            m.integrate(p, q)
    return m, params, pts, p12


class _Handle:
    """Owns a batch or server handle and what it uses."""

    def __init__(self, value, destroy, *keep):
        self.value, self._destroy, self._keep = value, destroy, keep

    def __del__(self):
        if self.value is not None:
            torch.cuda.synchronize()
            self._destroy(self.value)
            self.value = None


def _uneven(case):
    """Per-map cases of a batch or of served sessions: beams, azimuths and windows of the uneven batch workload."""
    rng = synth.SplitMix64(case["count"] * 7 + 3)
    pick = lambda v: v[int(rng.integers(1, 0, len(v))[0])]  # noqa: E731
    out = []
    for i in range(case["count"]):
        dims = pick([(256, 256, 256), (512, 512, 128)])
        out.append(dict(case, beams=pick([16, 32, 64, 128]), azimuths=pick([512, 1024, 2048]), dx=dims[0], dy=dims[1],
                        dz=dims[2], tau=max(case["tau"], 2 * case["voxel"]), kind="integrate"))
    return out


def _prepare_batch(case, seed):
    maps, pts, poses = [], [], []
    for i, c in enumerate(_uneven(case)):
        m, _, p, q = _map_in_use(c, seed * 64 + i, scans=2)
        maps.append(m)
        pts.append(p[-1])
        poses.append(q[-1])
    batch = b.tsdf_batch_create(len(maps))
    for _ in range(400):            # a long-running program is past the autotuner's trials
        b.tsdf_batch_integrate(batch, maps, pts, poses)
        b.tsdf_batch_sync(batch)
        if b.tsdf_batch_get_config(batch)["tuned"]:
            break
    return dict(batch=_Handle(batch, b.tsdf_batch_destroy, maps), maps=maps, pts=pts, poses=poses,
                grids=[_grid(m.handle, m.params, m) for m in maps])


def _prepare_serve(case, seed):
    pts, poses, params = [], [], []
    for i, c in enumerate(_uneven(case)):
        scene, tr = _scene_and_poses(c, seed * 64 + i, 1)
        gen = torch.Generator(device="cuda").manual_seed(seed * 64 + i)
        pts.append(_scan(c, scene, *tr[0], gen).cpu().pin_memory())
        poses.append(synth.pose12(*tr[0]))
        params.append(_params(c, tr[0][1]))
    most = max(p.shape[0] for p in pts)
    srv = _Handle(b.tsdf_server_create(64 << 30, max_points=most, max_batch=32, streams=2,
                                       max_outstanding=2 * len(pts), store_chunks=4096), b.tsdf_server_destroy)
    sessions = [b.tsdf_server_open_session(srv.value, p) for p in params]
    grids = [_grid(b.tsdf_server_session_map(srv.value, s), p, srv) for s, p in zip(sessions, params)]
    st = dict(server=srv, sessions=sessions, pts=pts, poses=poses, grids=grids)
    for _ in range(60):             # a server in service: its launch shapes are settled
        _serve(st)
    return st


def _register_field(case, scene, origin, seed):
    """A map's values and weights around the scene's surfaces (distance to the nearest one, in the map's
    fixed-point codes), as int16 arrays [z][y][x] on the GPU."""
    vs, tau = case["voxel"], float(np.float32(case["tau"]))
    ax = [(torch.arange(n, dtype=torch.float32, device="cuda") + o + 0.5) * vs
          for n, o in zip((case["dx"], case["dy"], case["dz"]), origin)]
    x, y, z = ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]
    dist = (z - scene.ground_z).expand(case["dz"], case["dy"], case["dx"]).clone()
    lo = [float(v[0]) - tau for v in ax]
    hi = [float(v[-1]) + tau for v in ax]
    for bx in scene.boxes:
        if any(bx[k] > hi[k] or bx[k + 3] < lo[k] for k in range(3)):
            continue
        q = [(a - 0.5 * (bx[k] + bx[k + 3])).abs() - 0.5 * (bx[k + 3] - bx[k]) for k, a in enumerate((x, y, z))]
        outside = (q[0].clamp_min(0) ** 2 + q[1].clamp_min(0) ** 2 + q[2].clamp_min(0) ** 2).sqrt()
        inside = torch.maximum(torch.maximum(q[0], q[1]), q[2]).clamp_max(0)
        dist = torch.minimum(dist, outside + inside)
    for cx, cy, rad, z0, z1 in scene.cylinders:
        if cx - rad > hi[0] or cx + rad < lo[0] or cy - rad > hi[1] or cy + rad < lo[1]:
            continue
        r = ((x - cx) ** 2 + (y - cy) ** 2).sqrt() - rad
        h = (z - 0.5 * (z0 + z1)).abs() - 0.5 * (z1 - z0)
        outside = (r.clamp_min(0) ** 2 + h.clamp_min(0) ** 2).sqrt()
        dist = torch.minimum(dist, outside + torch.maximum(r.expand_as(dist), h.expand_as(dist)).clamp_max(0))
    value = (dist.clamp(-tau, tau) * (32767.0 / tau)).round().to(torch.int16)
    gen = torch.Generator(device="cuda").manual_seed(seed + 5)
    weight = torch.randint(1, 65, dist.shape, generator=gen, device="cuda", dtype=torch.int16)
    weight[dist.abs() > tau] = 0
    value[weight == 0] = 0
    return value, weight


def _register_inputs(case, seed):
    scene, poses = _scene_and_poses(case, seed, 2)
    R, t = poses[-1]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    pts = _scan(case, scene, R, t, gen)
    params = _params(case, t)
    value, weight = _register_field(case, scene, params["origin"], seed)
    rng = synth.SplitMix64(seed + 9)
    w, v = rng.uniform(3, -0.01, 0.01), rng.uniform(3, -0.04, 0.04)    # an odometry guess: up to a degree and some cm off
    return params, value, weight, pts, synth.pose12(synth.rot_zyx(*w) @ R, t + v)


def _capacity(case):
    """Rows of the buffer that a program keeps for a map's triangles or points: room for all that its scans show."""
    voxels = case["dx"] * case["dy"] * case["dz"]
    return min(voxels // 4, 3500000) if case["kind"] == "mesh" else min(voxels // 8, 1000000)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return dict(_prepare_batch(case, seed), kind=kind)
    if kind == "serve":
        return dict(_prepare_serve(case, seed), kind=kind)
    if kind == "register":
        params, value, weight, pts, guess = _register_inputs(case, seed)
        m = b.TsdfMap(params)
        m.write(value.cpu().numpy(), weight.cpu().numpy())
        return dict(kind=kind, map=m, pts=pts, pose=guess)
    m, params, pts, poses = _map_in_use(case, seed, scans=6 if kind in ("mesh", "surface") else 3, dense=kind == "static")
    st = dict(kind=kind, map=m, pts=pts[-1], pose=poses[-1])
    if kind == "static":
        st["params"] = b.make_params(params)
        st["grid"] = torch.zeros(int(np.prod(params["dims"])), dtype=torch.int32, device="cuda")
        for p, q in zip(pts[:-1], poses[:-1]):
            b.tsdf_integrate_static(st["grid"], st["params"], p, p.shape[0], q, want_stats=False)
        return st
    st["grid"] = _grid(m.handle, params, m)
    if kind == "host":
        st["pts"] = st["pts"].cpu().pin_memory()
    elif kind == "drive":
        o = params["origin"]
        st["away"], st["home"] = (o[0] + case["step"], o[1] + 8, o[2]), o
        st["other"] = (pts[-2], poses[-2])
        _drive(st)
    elif kind in ("mesh", "surface"):
        m.integrate(pts[-1], poses[-1])
        row = (3, 3) if kind == "mesh" else (4,)
        st["out"] = torch.zeros((_capacity(case), *row), dtype=torch.float32, device="cuda")
        st["mine"] = torch.zeros_like(st["out"])
        st["odd"] = torch.randint(-2**62, 2**62, (math.prod(row),), device="cuda",
                                  generator=torch.Generator(device="cuda").manual_seed(1)) * 2 + 1
    return st


# ---------------------------------------------------------------- one pass

def _drive(st):
    m = st["map"]
    m.shift(st["away"])
    m.integrate(*st["other"])
    m.shift(st["home"])
    m.integrate(st["pts"], st["pose"])


def _serve(st):
    tickets = b.tsdf_server_submit_many(st["server"].value, st["sessions"], st["pts"], st["poses"])
    return b.tsdf_server_wait_many(st["server"].value, tickets)


def _ordered(st, n):
    """The first n triangles or points in an order of their own, in a buffer kept for them: the library's order is
    unspecified, and a program that compares, caches or stores them wants the same one each time. Ordered by a
    hash of their bits."""
    rows = st["out"].reshape(st["out"].shape[0], -1)[:n]
    order = torch.argsort((rows.view(torch.int32) * st["odd"]).sum(1))
    wide = (lambda v: v.view(torch.complex128).reshape(-1)) if rows.shape[1] == 4 else (lambda v: v)   # 16-byte rows move whole
    torch.index_select(wide(rows), 0, order, out=wide(st["mine"].reshape(st["mine"].shape[0], -1)[:rows.shape[0]]))
    return st["mine"]


def run(st):
    kind = st["kind"]
    if kind in ("integrate", "pool"):
        st["map"].integrate(st["pts"], st["pose"])
        return st["grid"]
    if kind == "host":
        st["map"].integrate_host(st["pts"], st["pose"])
        return dict(counters=st["map"].stats(), grid=st["grid"])
    if kind == "static":
        b.tsdf_integrate_static(st["grid"], st["params"], st["pts"], st["pts"].shape[0], st["pose"], want_stats=False)
        return st["grid"]
    if kind == "drive":
        _drive(st)
        return st["grid"]
    if kind == "batch":
        b.tsdf_batch_integrate(st["batch"].value, st["maps"], st["pts"], st["poses"])
        return st["grids"]
    if kind == "serve":
        return dict(counters=[r["stats"]["hits"] for r in _serve(st)], grids=st["grids"])
    if kind == "mesh":
        _, n = b.tsdf_extract_mesh(st["map"].handle, 1, st["out"])
        return dict(count=n, triangles=_ordered(st, n))
    if kind == "surface":
        _, n = b.tsdf_extract_surface(st["map"].handle, 1, st["out"])
        return dict(count=n, points=_ordered(st, n))
    if kind == "register":
        # the system at the guess (is it worth refining?), then the refinement
        first = b.tsdf_register_system(st["map"].handle, st["pts"], st["pose"])
        pose, res = b.tsdf_register(st["map"].handle, st["pts"], st["pose"], iterations=REGISTER_STEPS)
        return dict(first=first, pose=pose, rms=res["rms"], used=res["used_points"])
    raise ValueError(kind)


# ---------------------------------------------------------------- what a pass cannot do without

# Share of a scan's points whose march reaches the window, and how many of its samples fall into each
# touched voxel, as counted on the listed scenes.
_REACH = {"room": 0.98, "outdoor": 0.25, "corridor": 0.55}
_SHARED = {"room": 1.6, "outdoor": 1.8, "corridor": 2.65}


def _scan_work(c):
    """Points read once, touched voxels read and written once; about 30 operations per march sample."""
    n = c["beams"] * c["azimuths"]
    steps = 2 * math.floor(c["tau"] / c["voxel"] + 1e-9) + 1
    inside = min(1.0, c["dx"] * c["voxel"] / 32.0) if c["scene"] == "outdoor" else 1.0
    reach = {"room": 5.0, "outdoor": 12.0 * inside, "corridor": 4.0}[c["scene"]]
    fill = 1 + 2 * math.floor(math.tan(math.radians(_VFOV[c["scene"]] / c["beams"])) * reach / c["voxel"])
    samples = n * _REACH[c["scene"]] * inside * steps * fill
    touched = min(samples / _SHARED[c["scene"]], 0.25 * c["dx"] * c["dy"] * c["dz"])
    return 16.0 * n + 8.0 * touched, 30.0 * samples


def work(case):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        parts = [_scan_work(c) for c in _uneven(case)]
        return dict(bytes=sum(p[0] for p in parts), flops=sum(p[1] for p in parts))
    bytes_, flops = _scan_work(case)
    voxels = float(case["dx"] * case["dy"] * case["dz"])
    n = float(case["beams"] * case["azimuths"])
    if kind == "drive":
        # two scans, and two shifts that each move the bricks of the layers that leave and enter
        moved = voxels * (1 - (1 - case["step"] / case["dx"]) * (1 - 8 / case["dy"]))
        return dict(bytes=2 * bytes_ + 2 * 4 * 2 * moved, flops=2 * flops)
    if kind in ("mesh", "surface"):
        # the window read once, and what lies on its surfaces written: crossings and triangles per touched voxel
        # of a scan, as counted on the listed scene
        out = (bytes_ - 16.0 * n) / 8.0 * (2.5 * 36.0 if kind == "mesh" else 0.45 * 16.0)
        return dict(bytes=4.0 * voxels + out, flops=40.0 * n)
    if kind == "register":
        evals = REGISTER_STEPS + 1
        return dict(bytes=n * (16.0 + 32.0), flops=evals * 200.0 * n)
    return dict(bytes=bytes_, flops=flops)


# ---------------------------------------------------------------- in 64 bits

def _exact_system(case, params, value, weight, pts, pose):
    """Normal equations of scan-to-map registration in binary64 (see tsdf_register_system): the 29 sums."""
    o = torch.tensor(params["origin"], device="cuda")
    dims = torch.tensor(params["dims"], device="cuda")
    T = torch.tensor(np.asarray(pose, np.float64).reshape(3, 4), device="cuda")
    p = pts[torch.isfinite(pts).all(1), :3].double()
    q = (p[:, None, :] * T[None, :, :3]).sum(2) + T[:, 3]
    u = q / params["voxel_size"] - 0.5
    i0 = torch.floor(u).long()
    f = u - i0
    rel = i0 - o
    ok = ((rel >= 0) & (rel + 1 < dims)).all(1)
    q, f, rel = q[ok], f[ok], rel[ok]
    c, keep = {}, torch.ones(q.shape[0], dtype=torch.bool, device="cuda")
    for k in range(8):
        ix = rel + torch.tensor([k & 1, (k >> 1) & 1, k >> 2], device="cuda")
        at = (ix[:, 2] * params["dims"][1] + ix[:, 1]) * params["dims"][0] + ix[:, 0]
        c[k] = value.reshape(-1)[at].double() * (params["tau"] / 32767.0)
        keep &= weight.reshape(-1)[at] >= 1
    fx, fy, fz = f.unbind(1)
    w = [(1 - fx, fx), (1 - fy, fy), (1 - fz, fz)]
    d = sum(c[k] * w[0][k & 1] * w[1][(k >> 1) & 1] * w[2][k >> 2] for k in range(8))
    keep &= d.abs() < params["tau"]
    g = []
    for a in range(3):
        e, s = [x for x in range(3) if x != a], 1 << a
        g.append(sum((c[k | s] - c[k]) * w[e[0]][(k >> e[0]) & 1] * w[e[1]][(k >> e[1]) & 1]
                     for k in range(8) if not k & s) / params["voxel_size"])
    g = torch.stack(g, 1)
    J = torch.cat([torch.linalg.cross(q, g), g], 1)[keep]
    d = d[keep]
    H, grad = (J[:, :, None] * J[:, None, :]).sum(0).cpu().numpy(), (J * d[:, None]).sum(0).cpu().numpy()
    return H, grad, float((d * d).sum()), int(keep.sum())


def _exact_register(case, seed):
    params, value, weight, pts, pose = _register_inputs(case, seed)
    T = np.asarray(pose, np.float64).reshape(3, 4).copy()
    first, rms = None, None
    for _ in range(REGISTER_STEPS):
        H, g, cost, used = _exact_system(case, params, value, weight, pts, T)
        if first is None:
            first = np.concatenate([H[np.triu_indices(6)], g, [cost, float(used)]])
        rms = math.sqrt(cost / used)
        xi = np.linalg.solve(H, -g)
        th = np.linalg.norm(xi[:3])
        K = np.array([[0, -xi[2], xi[1]], [xi[2], 0, -xi[0]], [-xi[1], xi[0], 0]])
        E = np.eye(3) + (math.sin(th) / th if th > 1e-12 else 1.0) * K + ((1 - math.cos(th)) / th**2 if th > 1e-12 else 0.0) * K @ K
        T = np.concatenate([E @ T[:, :3], (E @ T[:, 3] + xi[3:])[:, None]], 1)
    return dict(first=first, pose=T.reshape(12), rms=rms, used=None)


def exact(case, seed):
    # Grids and counters are whole numbers. Triangles and points are single IEEE operations on them, in an
    # order that has no 64-bit counterpart.
    return _exact_register(case, seed) if case["kind"] == "register" else None
