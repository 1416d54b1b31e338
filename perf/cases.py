"""Performance cases: what a mapping program has this framework do, call by call.

A mapper keeps a voxel map on the GPU, integrates scan after scan into it and
looks voxels up around the sensor; a calibration or odometry program
differentiates a frame; a fleet server integrates a scan for each of many maps
in one step.  Each case is one such pass through the public entry points, on
the sensors, scenes and map parameters of this repository's workloads
(workloads.py, synth.py), over their range of sizes.

listed() and draw(rng) give cases, prepare(case, seed) what the program holds
before the call, run(state) one pass, work(case) the bytes and operations a
pass cannot do without, and exact(case, seed) what the first pass returns in
64-bit arithmetic.
"""
import math

import numpy as np
import torch

from paper_2206_06079_gb300 import ohm, synth, workloads as W

FRAC = 16
U = 1 << FRAC
LAYERS = {"occ": W.OCC, "ndt": W.NDT, "tsdf": W.TSDF, "counts": W.COUNTS, "decay": W.DECAY, "mean": W.MEAN}


def listed():
    return [
        # one packet of a 16-beam lidar, integrated as it arrives; the program
        # waits for each (the default, blocking call)
        dict(name="packet_room", kind="scan", scene="room", beams=16, azimuths=24, voxel=0.1, range=20.0,
             layers="occ", ring=3, wait=True, window=16, landmarks=500),
        # the repository's room scan: 32,768 rays, occupancy, blocking call
        dict(name="scan_room", kind="scan", scene="sphere", beams=1, azimuths=32768, voxel=0.1, range=20.0,
             layers="occ", ring=3, wait=True, window=32, landmarks=4096),
        # a driving lidar at 131,072 rays, occupancy + NDT-OM, scans enqueued
        # back to back: the repository's tunnel workload, in a mapped tunnel
        dict(name="drive_tunnel", kind="scan", scene="tunnel", beams=128, azimuths=1024, voxel=0.1, range=50.0,
             layers="occ+ndt", ring=3, wait=False, window=64, landmarks=16384),
        # the largest scan: 262,144 rays into 5 cm voxels
        dict(name="drive_fine", kind="scan", scene="tunnel", beams=128, azimuths=2048, voxel=0.05, range=20.0,
             layers="occ", ring=2, wait=False, window=64, landmarks=16384),
        # survey mapping with every per-voxel statistic, an odd azimuth count
        dict(name="survey_layers", kind="scan", scene="tunnel", beams=64, azimuths=1021, voxel=0.1, range=20.0,
             layers="occ+ndt+counts+decay+mean", ring=3, wait=False, window=32, landmarks=8192),
        # unknown space: a new map built from an outdoor drive, then looked up
        dict(name="explore_outdoor", kind="build", scans=24, beams=128, azimuths=1024, voxel=0.1, range=30.0,
             layers="occ+ndt", regions=8192, ndt_regions=2048, window=128, landmarks=16384),
        # a depth camera's TSDF, frame by frame
        dict(name="depth_tsdf", kind="depth", width=640, height=480, voxel=0.05, trunc=0.2, layers="tsdf", ring=3,
             stride=4),
        # training or calibration through a depth frame: forward and backward
        dict(name="grad_tsdf", kind="tsdf_grad", width=640, height=480, voxel=0.05, trunc=0.2, queries=20000),
        # pose and point gradients of NDT statistics: forward and backward
        dict(name="grad_ndt", kind="ndt_grad", beams=64, azimuths=1024, voxel=0.1, range=50.0, queries=20000),
        # a fleet: one scan of mixed sensors for each of 16 maps in one step
        dict(name="fleet_16", kind="fleet", maps=16, window=48, landmarks=2048),
        # a map published whole: every region's layers exported, and a lookup
        dict(name="publish_room", kind="publish", beams=1, azimuths=131072, voxel=0.05, range=20.0,
             layers="occ+ndt+counts", window=64, landmarks=16384),
        # per-frame counting into a dense local grid inside a real-time loop
        dict(name="count_grid", kind="count", rays=30011, voxel=0.1, range=12.0, nx=112, ny=96, nz=56),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["scan"] * 5 + ["build", "depth", "depth", "tsdf_grad", "ndt_grad", "fleet", "publish", "count"])
    if kind == "scan":
        scene = rng.choice(["room", "sphere", "tunnel", "tunnel"])
        rays = _log(rng, 300, 262144)
        beams = 1 if scene == "sphere" else min(rng.choice([16, 32, 64, 128, 53]), max(1, rays // 8))
        layers = rng.choice(["occ", "occ", "occ+ndt", "occ+ndt", "occ+counts", "occ+mean", "occ+ndt+counts+decay+mean"])
        small = layers.startswith("occ+ndt+counts")
        rng_m = rng.choice([20.0, 30.0, 50.0] if scene == "tunnel" else [12.0, 20.0])
        voxel = 0.1 if small or rng_m > 20.0 else rng.choice([0.1, 0.05, 0.08])
        rays = min(rays, 131072) if small or rng_m > 20.0 else rays
        return dict(kind=kind, scene=scene, beams=beams, azimuths=max(1, rays // beams), voxel=voxel, range=rng_m,
                    layers=layers, ring=rng.choice([2, 3]), wait=rng.random() < 0.4, window=rng.choice([16, 24, 32, 64]),
                    landmarks=_log(rng, 100, 16384))
    if kind == "build":
        return dict(kind=kind, scans=rng.randint(4, 24), beams=rng.choice([16, 32, 64, 128]), azimuths=_log(rng, 300, 1024),
                    voxel=0.1, range=rng.choice([20.0, 30.0]), layers=rng.choice(["occ", "occ+ndt"]), regions=8192,
                    ndt_regions=2048, window=32, landmarks=_log(rng, 500, 16384))
    if kind in ("depth", "tsdf_grad"):
        w = _log(rng, 80, 640)
        h = max(40, min(480, int(w * rng.choice([0.5, 0.566, 0.75]))))
        c = dict(kind=kind, width=w, height=h, voxel=rng.choice([0.05, 0.05, 0.04, 0.1]), trunc=rng.choice([0.1, 0.2]))
        if kind == "depth":
            c.update(layers=rng.choice(["tsdf", "tsdf", "occ+tsdf"]), ring=rng.choice([2, 3]), stride=rng.choice([2, 3, 4]))
        else:
            c.update(queries=_log(rng, 500, 20000))
        return c
    if kind == "ndt_grad":
        return dict(kind=kind, beams=rng.choice([16, 32, 64, 128]), azimuths=_log(rng, 100, 1024), voxel=0.1,
                    range=rng.choice([20.0, 50.0]), queries=_log(rng, 500, 20000))
    if kind == "fleet":
        return dict(kind=kind, maps=rng.randint(2, 16), window=rng.choice([16, 32, 48]), landmarks=_log(rng, 200, 2048))
    if kind == "publish":
        return dict(kind=kind, beams=1, azimuths=_log(rng, 2000, 131072), voxel=rng.choice([0.05, 0.1]), range=20.0,
                    layers=rng.choice(["occ", "occ+counts", "occ+ndt"]), window=rng.choice([32, 64]),
                    landmarks=_log(rng, 500, 16384))
    return dict(kind=kind, rays=_log(rng, 500, 32768), voxel=rng.choice([0.1, 0.08]), range=12.0, nx=rng.randint(40, 120),
                ny=rng.randint(40, 120), nz=rng.randint(20, 60))


# ---------------------------------------------------------------------------
# Inputs.
# ---------------------------------------------------------------------------
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _layer_bits(text):
    bits = 0
    for name in text.split("+"):
        bits |= LAYERS[name]
    return bits


def _scan(case, seed, k):
    """Scan k of a case's sensor: the pose moves with k, the noise is new."""
    scene, dev = case["scene"], _dev()
    n = case["beams"] * case["azimuths"]
    if scene == "sphere":
        return synth.room_scan(seed=seed * 31 + k, n=n, device=dev,
                               sensor=(0.3 * math.sin(seed + 2.0 * k), 0.3 * math.cos(seed + 2.0 * k), 1.0))
    if scene == "room":
        return _room_sweep(case["beams"], case["azimuths"], seed * 31 + k)
    i = (seed * 37 + k) % 100
    return synth.tunnel_scan(i, seed=seed % 100003 + 1, beams=case["beams"], azimuths=case["azimuths"], max_range=case["range"],
                             device=dev)


def _room_sweep(beams, azimuths, seed):
    """Part of a spinning lidar's sweep of the box room: `azimuths` steps of
    0.2 degrees from a seeded heading, closed-form walls."""
    dev = _dev()
    g = torch.Generator().manual_seed(int(seed))
    r = torch.rand(4, generator=g, dtype=torch.float64)
    d = synth.lidar_directions(beams, azimuths, 15.0, dtype=torch.float64)
    el = torch.asin(d[:, 2])
    az = 2 * math.pi * r[0] + (torch.arange(beams * azimuths, dtype=torch.float64) % azimuths) * math.radians(0.2)
    u = torch.stack([torch.cos(el) * torch.cos(az), torch.cos(el) * torch.sin(az), torch.sin(el)], 1).to(dev)
    o = torch.tensor([float(r[1]) - 0.5, float(r[2]) - 0.5, 1.0 + 0.2 * float(r[3])], dtype=torch.float64, device=dev)
    lo = torch.tensor(synth.ROOM_MIN, dtype=torch.float64, device=dev)
    hi = torch.tensor(synth.ROOM_MAX, dtype=torch.float64, device=dev)
    safe = torch.where(u == 0, torch.full_like(u, 1e-12), u)
    t = (torch.where(u > 0, hi, lo) - o).div(safe).min(1).values
    t = t + (torch.randn(u.shape[0], generator=g, dtype=torch.float64) * 0.02).to(dev)
    return synth.RaySet(o[None].float(), (o + t[:, None] * u).float(), torch.zeros(u.shape[0], dtype=torch.uint8, device=dev))


def _outdoor(case, seed):
    """A drive of case["scans"] scans about 2 m apart through the outdoor world."""
    world = synth.world_scene(seed=0x0A16 + seed % 7)
    robot, t0 = seed % 8, float(seed % 500)
    kind = "lidar%dx%d" % (case["beams"], case["azimuths"])
    return [synth.world_scan(world, robot, t0 + 2.0 * k, kind, device=_dev(), max_range=case["range"], seed=seed + k)
            for k in range(case["scans"])]


def _points(case, ray):
    """Lookup points of a pass: a box of voxel centres around the sensor
    (window x window x window / 4, a local planner's grid) and some of the
    scan's end points."""
    dev, w, v = ray.endpoints.device, case["window"], case["voxel"]
    ax = (torch.arange(w, dtype=torch.float64, device=dev) - w // 2 + 0.5) * v
    az = (torch.arange(max(1, w // 4), dtype=torch.float64, device=dev) - w // 8 + 0.5) * v
    base = torch.floor(ray.origins[0].double() / v) * v
    box = torch.stack(torch.meshgrid(ax, ax, az, indexing="ij"), -1).reshape(-1, 3) + base
    n = ray.endpoints.shape[0]
    at = torch.linspace(0, n - 1, min(n, case["landmarks"]), dtype=torch.float64, device=dev).long()
    return torch.cat([box.float(), ray.endpoints[at]]).contiguous()


def _map_params(case, n, regions, ndt_regions=1024):
    return dict(voxel_size=case["voxel"], layers=_layer_bits(case["layers"]), max_range=case["range"], hit=W.HIT, miss=W.MISS,
                max_rays=n, max_regions=regions, max_ndt_regions=min(ndt_regions, regions))


def _pool(case):
    """Region pool of a scan case: what its trajectory can touch, with room."""
    per_m = 1.0 / (32 * case["voxel"])
    if case["scene"] in ("room", "sphere"):
        side = 2 * 7.0 * per_m + 3
        return int(min(4096, side * side * (6.0 * per_m + 3)))
    r = case["range"] + 2.0
    h = 0.45 * r * per_m * 2 + 3
    return int(min(24576, (2 * r * per_m + 3) ** 2 * h * 0.7 + 512))


def _lookup_layers(case):
    names = case["layers"].split("+")
    return dict(ndt="ndt" in names, counts="counts" in names, path_sum="decay" in names, mean="mean" in names, tsdf="tsdf" in names)


_FLEET_KINDS = ("lidar16x1800", "lidar64x1024", "lidar128x2048", "depth424x240")


def _fleet(case, seed):
    """Per map of the fleet: (map parameters, scan, lookup points)."""
    out = []
    for i in range(case["maps"]):
        scene, voxel = ("tunnel", "room")[i % 2], (0.1, 0.05)[(i // 2) % 2]
        kind = _FLEET_KINDS[(seed * 7 + i * 5 + i // 4) % 4]
        ray = synth.mixed_scan(scene, kind, seed * 64 + i, device=_dev())
        p = dict(W.room_params(), voxel_size=voxel, max_range=20.0, max_rays=128 * 2048,
                 max_regions=6144 if voxel == 0.05 and scene == "tunnel" else 2048)
        out.append((p, ray, _points(dict(case, voxel=voxel), ray)))
    return out


def _depth(case, seed, k):
    """Depth frame k: image, intrinsics, pose (3 x 4)."""
    w, h, s = case["width"], case["height"], case["width"] / 640.0
    K = (525.0 * s, 525.0 * s, (w - 1) / 2.0, (h - 1) / 2.0)
    scene = synth.depth_scene(seed=0x0A14 + seed % 5)
    depth, pos, R = synth.depth_frame(scene, (seed + 3 * k) % 64, width=w, height=h, fx=K[0], fy=K[1], cx=K[2], cy=K[3],
                                      device=_dev())
    g = torch.Generator().manual_seed(seed * 31 + k)
    depth = depth + (0.002 * torch.randn(h, w, generator=g)).to(depth.device)  # sensor noise
    return depth, K, np.concatenate([R.numpy(), pos.numpy()[:, None]], 1)


def _surface_points(depth, K, pose, stride, z_min=0.3, z_max=6.0):
    """Points at, before and behind the surface seen by every stride-th pixel."""
    h, w = depth.shape
    dev = depth.device
    vv, uu = torch.meshgrid(torch.arange(0, h, stride, device=dev), torch.arange(0, w, stride, device=dev), indexing="ij")
    z = depth[vv, uu].double()
    z = torch.where((z > z_min) & (z <= z_max), z, torch.full_like(z, 1.0)) + ((uu + vv) % 5 - 2).double() * 0.03
    pc = torch.stack([(uu - K[2]) / K[0] * z, (vv - K[3]) / K[1] * z, z], -1).reshape(-1, 3)
    P = torch.from_numpy(pose).to(dev)
    return (pc @ P[:, :3].T + P[:, 3]).float().contiguous()


def _tsdf_map(case, n):
    per = 32 * case["voxel"]
    regions = int((8.0 / per + 2) ** 2 * (5.0 / per + 2))
    return dict(W.tsdf_params(), voxel_size=case["voxel"], tsdf_trunc=case["trunc"], layers=_layer_bits(case.get("layers", "tsdf")),
                max_rays=n, max_regions=max(256, min(4096, regions)))


def _grad_inputs(case, seed):
    """What the two adjoint cases differentiate."""
    dev = _dev()
    g = torch.Generator().manual_seed(seed * 13 + 5)
    if case["kind"] == "tsdf_grad":
        depth, K, pose = _depth(case, seed, 0)
        stride = max(1, int(math.sqrt(case["width"] * case["height"] / case["queries"])))
        pts = _surface_points(depth, K, pose, stride)[: case["queries"]]
        return depth, K, pose, pts, torch.randn(pts.shape[0], generator=g).to(dev)
    ray = _scan(dict(case, scene="tunnel"), seed, 0)
    yaw = 0.3 + 0.01 * (seed % 50)
    c, s = math.cos(yaw), math.sin(yaw)
    pose = np.array([[c, -s, 0, 1.5], [s, c, 0, -0.5], [0, 0, 1, 0.25]])
    q = min(case["queries"], ray.endpoints.shape[0])
    at = torch.linspace(0, ray.endpoints.shape[0] - 1, q, dtype=torch.float64, device=dev).long()
    P = torch.from_numpy(pose).to(dev)
    pts = (ray.endpoints[at].double() @ P[:, :3].T + P[:, 3]).float().contiguous()
    return ray, pose, pts, torch.randn(q, 3, generator=g).to(dev), torch.randn(q, 6, generator=g).to(dev)


_PUBLISH_BOX = ((-4, 4), (-3, 3), (-1, 3))  # regions of 1.6 m (5 cm voxels) that hold the box room


def _publish_box(case):
    s = 0.05 / case["voxel"]
    return [(int(math.floor(lo * s)), int(math.ceil(hi * s))) for lo, hi in _PUBLISH_BOX]


def _first_rays(case):
    """One short pass-through ray in each region of the published box, in a
    fixed order, so that the regions' export order is the same in every run."""
    size = 32 * case["voxel"]
    (x0, x1), (y0, y1), (z0, z1) = _publish_box(case)
    return [torch.tensor([[(x + 0.51) * size, (y + 0.51) * size, (z + 0.51) * size]], dtype=torch.float32)
            for z in range(z0, z1) for y in range(y0, y1) for x in range(x0, x1)]


def _publish_scan(case, seed):
    """A room scan that stays inside the published box."""
    return synth.room_scan(seed=seed, n=case["azimuths"], device=_dev(), room_min=(-5.0, -4.0, -0.4), room_max=(5.0, 4.0, 3.6),
                           sensor=(0.4 * math.sin(seed), 0.4 * math.cos(seed), 1.0))


# ---------------------------------------------------------------------------
# State and passes.
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind, case=case, passes=0)
    if kind == "scan":
        st["ring"] = [_scan(case, seed, k) for k in range(case["ring"])]
        st["points"] = _points(case, st["ring"][0])
        st["map"] = ohm.Map(**_map_params(case, st["ring"][0].n, _pool(case)))
        for r in st["ring"][1:]:  # the place has been seen before
            st["map"].integrate(r.origins, r.endpoints, r.flags)
    elif kind == "build":
        st["scans"] = _outdoor(case, seed)
        st["points"] = _points(case, st["scans"][-1])
    elif kind == "depth":
        st["frames"] = [_depth(case, seed, k) for k in range(case["ring"])]
        st["points"] = _surface_points(*st["frames"][0], case["stride"])
        st["map"] = ohm.Map(**_tsdf_map(case, case["width"] * case["height"]))
        for d, K, pose in st["frames"][1:]:
            st["map"].integrate_depth(d, K, pose)
    elif kind == "tsdf_grad":
        depth, st["K"], st["pose"], st["points"], st["grad"] = _grad_inputs(case, seed)
        st["depth"] = depth.requires_grad_(True)
        st["xi"] = torch.zeros(6, dtype=torch.float64, requires_grad=True)
        st["map"] = ohm.Map(**_tsdf_map(case, depth.numel()))
    elif kind == "ndt_grad":
        st["ray"], st["pose"], st["points"], st["gmean"], st["gcov"] = _grad_inputs(case, seed)
        st["endpoints"] = st["ray"].endpoints.requires_grad_(True)
        st["xi"] = torch.zeros(6, dtype=torch.float64, requires_grad=True)
        c = dict(case, layers="occ+ndt", scene="tunnel")
        st["map"] = ohm.Map(**_map_params(c, st["ray"].n, _pool(c)))
    elif kind == "fleet":
        fleet = _fleet(case, seed)
        st["maps"] = [ohm.Map(**p) for p, _, _ in fleet]
        st["batch"] = ohm.Batch(st["maps"])
        st["raysets"] = [(r.origins, r.endpoints, r.flags) for _, r, _ in fleet]
        st["points"] = [p for _, _, p in fleet]
        st["stream"] = torch.cuda.Stream()
        torch.cuda.synchronize()
    elif kind == "publish":
        ray = _publish_scan(case, seed)
        st["points"] = _points(case, ray)
        first = _first_rays(case)
        st["map"] = ohm.Map(**_map_params(case, max(ray.n, 1), len(first) + 64))
        for p in first:
            st["map"].integrate(p, p, np.array([1], np.uint8))
        st["map"].integrate(ray.origins, ray.endpoints, ray.flags)
        st["regions"] = len(first)
    else:
        ray = synth.room_scan(seed=seed, n=case["rays"], device=_dev())
        st["ray"] = ray
        dims = (case["nx"], case["ny"], case["nz"])
        st["grid"] = dict(voxel_size=case["voxel"], max_range=case["range"], corner=(-dims[0] // 2, -dims[1] // 2, -5), dims=dims)
        n = dims[0] * dims[1] * dims[2]
        st["hits"] = torch.zeros(n, dtype=torch.int32, device=_dev())
        st["misses"] = torch.zeros(n, dtype=torch.int32, device=_dev())
    return st


def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "scan":
        r = st["ring"][st["passes"] % len(st["ring"])]
        st["passes"] += 1
        st["map"].integrate(r.origins, r.endpoints, r.flags, sync=case["wait"])
        return st["map"].query(st["points"], **_lookup_layers(case))
    if kind == "build":
        first = st["scans"][0]
        with ohm.Map(**_map_params(case, first.n, case["regions"], case["ndt_regions"])) as m:
            for r in st["scans"]:
                m.integrate(r.origins, r.endpoints, r.flags, sync=False)
            m.sync()
            return m.query(st["points"], **_lookup_layers(case))
    if kind == "depth":
        d, K, pose = st["frames"][st["passes"] % len(st["frames"])]
        st["passes"] += 1
        st["map"].integrate_depth(d, K, pose, sync=False)
        return st["map"].query(st["points"], **_lookup_layers(case))
    if kind == "tsdf_grad":
        D = ohm.TsdfFrame.apply(st["depth"], st["xi"], st["map"], st["K"], st["pose"], st["points"])
        gd, gx = torch.autograd.grad(D, (st["depth"], st["xi"]), st["grad"])
        return dict(distance=D.detach(), grad_depth=gd, grad_twist=gx)
    if kind == "ndt_grad":
        mean, cov = ohm.NdtFrame.apply(st["endpoints"], st["xi"], st["map"], st["pose"], st["ray"].origins, st["ray"].flags,
                                       st["points"])
        ge, gx = torch.autograd.grad((mean, cov), (st["endpoints"], st["xi"]), (st["gmean"], st["gcov"]))
        return dict(mean=mean.detach(), cov=cov.detach(), grad_endpoints=ge, grad_twist=gx)
    if kind == "fleet":
        with torch.cuda.stream(st["stream"]):
            st["batch"].integrate(st["raysets"])
            out = [m.query(p) for m, p in zip(st["maps"], st["points"])]
        return dict(occupancy=[q["occupancy"] for q in out], known=[q["known"] for q in out])
    if kind == "publish":
        look = _lookup_layers(case)
        out = st["map"].export(counts=look["counts"], ndt=look["ndt"], count=st["regions"])
        return dict(map=out, around=st["map"].query(st["points"], ndt=look["ndt"], counts=look["counts"]))
    ray = st["ray"]
    st["hits"].zero_()
    st["misses"].zero_()
    ohm.count_rays_noalloc(st["grid"], ray.origins, ray.endpoints, ray.flags, st["hits"], st["misses"])
    return dict(hits=st["hits"], misses=st["misses"])


# ---------------------------------------------------------------------------
# Work that a pass cannot do without.
# ---------------------------------------------------------------------------
def _walk_work(n, length, voxel, solid_angle):
    """(voxel visits, distinct voxels) of n rays of mean length `length` from
    one sensor: near it rays share voxels (a shell of radius r holds
    solid_angle r^2 / v^2 of them per voxel of depth), further out each ray has
    its own.  A ray crosses about 1.5 voxels per voxel length."""
    visits = 1.5 * n * length / voxel + n
    shared = voxel * math.sqrt(1.5 * n / solid_angle)
    if shared >= length:
        return visits, solid_angle * length ** 3 / (3 * voxel ** 3)
    return visits, solid_angle * shared ** 3 / (3 * voxel ** 3) + 1.5 * n * (length - shared) / voxel


def _scan_length(scene, rng):
    """(mean ray length, solid angle) of a scene's scans, from the scenes' sizes."""
    if scene == "sphere":
        return min(rng, 3.5), 4 * math.pi
    if scene == "room":
        return min(rng, 5.0), 0.25 * 4 * math.pi
    if scene == "outdoor":
        return 0.6 * rng, 0.38 * 4 * math.pi
    return 5.5 + 0.1 * rng + (0.02 * rng if rng > 20 else 0.0), 0.38 * 4 * math.pi


def work(case):
    kind = case["kind"]
    layers = case.get("layers", "occ").split("+")
    per_voxel = 8 + (16 if "counts" in layers else 0) + (16 if "decay" in layers else 0)
    per_sample = 8 + (160 if "ndt" in layers else 0) + (16 if "mean" in layers else 0)
    per_point = 12 + 5 + 4 + (40 + 80 if "ndt" in layers else 0) + (16 if "counts" in layers else 0)
    points = case.get("window", 0) ** 2 * max(1, case.get("window", 0) // 4) + case.get("landmarks", 0)

    def scan(n, scene, rng, voxel):
        length, angle = _scan_length(scene, rng)
        visits, voxels = _walk_work(n, length, voxel, angle)
        return 13 * n + per_voxel * voxels + per_sample * 0.5 * n, 12 * visits

    if kind == "scan":
        b, f = scan(case["beams"] * case["azimuths"], case["scene"], case["range"], case["voxel"])
        return dict(bytes=b + per_point * points, flops=f)
    if kind == "build":
        b, f = scan(case["beams"] * case["azimuths"], "outdoor", case["range"], case["voxel"])
        return dict(bytes=case["scans"] * b + per_point * points, flops=case["scans"] * f)
    if kind in ("depth", "tsdf_grad"):
        n = case["width"] * case["height"]
        visits = n * (1.5 * 2 * case["trunc"] / case["voxel"] + 1)
        voxels = min(visits, 60.0 / case["voxel"] ** 2 * (2 * case["trunc"] / case["voxel"] + 1) * 0.5)
        if kind == "depth":
            return dict(bytes=4 * n + 16 * voxels + 20 * n / case["stride"] ** 2, flops=20 * visits)
        return dict(bytes=12 * n + 24 * voxels + 24 * case["queries"], flops=45 * visits)
    if kind == "ndt_grad":
        layers, n = ["occ", "ndt"], case["beams"] * case["azimuths"]
        per_sample = 168
        b, f = scan(n, "tunnel", case["range"], case["voxel"])
        return dict(bytes=b + (13 + 12 + 80) * n + 130 * case["queries"], flops=f + 80 * n)
    if kind == "fleet":
        rays = (16 * 1800, 64 * 1024, 128 * 2048, 424 * 240)
        b = f = 0.0
        for i in range(case["maps"]):
            bb, ff = scan(sum(rays) / 4, ("tunnel", "room")[i % 2], 20.0, (0.1, 0.05)[(i // 2) % 2])
            b, f = b + bb + per_point * points, f + ff
        return dict(bytes=b, flops=f)
    if kind == "publish":
        regions = 1
        for lo, hi in _publish_box(case):
            regions *= hi - lo
        per = 2 * (4 + (8 if "counts" in layers else 0) + (80 if "ndt" in layers else 0))
        return dict(bytes=regions * 32768 * per + per_point * points, flops=regions * 32768)
    visits, _ = _walk_work(case["rays"], 3.5, case["voxel"], 4 * math.pi)
    return dict(bytes=13 * case["rays"] + 8 * case["nx"] * case["ny"] * case["nz"], flops=12 * visits)


# ---------------------------------------------------------------------------
# The same results in 64 bits, in plain torch: an integer voxel walk over all
# rays at once, and per-voxel updates as sums.
# ---------------------------------------------------------------------------
_BIAS = 1 << 20


def _quantise(x, voxel):
    return torch.round(x.double() * (float(U) / voxel)).long()


def _pack(v):
    return ((v[..., 0] + _BIAS) << 42) | ((v[..., 1] + _BIAS) << 21) | (v[..., 2] + _BIAS)


def _walk(a, b):
    """Voxel walk of every ray from a to b (fixed point): (voxels visited in
    order as (m, 3), ray of each, is each the ray's last)."""
    delta = b - a
    A, neg = delta.abs(), delta < 0
    va, vb = a >> FRAC, b >> FRAC
    n = (vb - va).abs()
    order = torch.argsort(n.sum(1), descending=True)
    A, neg, va, n = A[order], neg[order], va[order], n[order]
    d0 = torch.where(neg, a[order] - va * U, (va + 1) * U - a[order])
    step = torch.where(neg, -1, 1)
    cxy = d0[:, 0] * A[:, 1] - d0[:, 1] * A[:, 0]
    cxz = d0[:, 0] * A[:, 2] - d0[:, 2] * A[:, 0]
    cyz = d0[:, 1] * A[:, 2] - d0[:, 2] * A[:, 1]
    total = n.sum(1)
    at = torch.cumsum(total + 1, 0) - (total + 1)
    out = torch.empty((int((total + 1).sum()), 3), dtype=torch.int32, device=a.device)
    steps = torch.bincount(total.cpu(), minlength=1).numpy()
    alive = np.cumsum(steps[::-1])[::-1]  # alive[i]: rays with at least i steps
    v, left = va.clone(), n.clone()
    for i in range(len(steps)):
        m = int(alive[i])
        out[at[:m] + i] = v[:m].int()
        if i + 1 >= len(steps):
            break
        m = int(alive[i + 1])
        if m == 0:
            break
        x, y, z = cxy[:m], cxz[:m], cyz[:m]
        l = left[:m]
        bx = (x < 0) & (y < 0)
        by = ~bx & (x >= 0) & (z < 0)
        bz = ~bx & ~by
        none = torch.where(bx, l[:, 0], torch.where(by, l[:, 1], l[:, 2])) == 0
        lz, ly = l[:, 2] > 0, l[:, 1] > 0
        bz = torch.where(none, lz, bz)
        by = torch.where(none, ~lz & ly, by)
        bx = ~bz & ~by
        sel = torch.stack([bx, by, bz], 1).long()
        AU = A[:m] * U
        cxy[:m] += sel[:, 0] * AU[:, 1] - sel[:, 1] * AU[:, 0]
        cxz[:m] += sel[:, 0] * AU[:, 2] - sel[:, 2] * AU[:, 0]
        cyz[:m] += sel[:, 1] * AU[:, 2] - sel[:, 2] * AU[:, 1]
        v[:m] += sel * step[:m]
        left[:m] -= sel
    ray = torch.repeat_interleave(order, total + 1)
    last = torch.zeros(out.shape[0], dtype=torch.bool, device=a.device)
    last[at + total] = True
    return out, ray, last


class _Table:
    """Per-voxel columns over a sorted key list."""

    def __init__(self, dev):
        self.keys = torch.empty(0, dtype=torch.long, device=dev)
        self.col = {}

    def add(self, keys):
        merged = torch.unique(torch.cat([self.keys, keys]))
        at = torch.searchsorted(merged, self.keys)
        for name, (old, empty) in list(self.col.items()):
            new = torch.full((merged.shape[0],) + old.shape[1:], empty, dtype=old.dtype, device=old.device)
            new[at] = old
            self.col[name] = (new, empty)
        self.keys = merged

    def column(self, name, empty, dtype, width=()):
        if name not in self.col:
            self.col[name] = (torch.full((self.keys.shape[0],) + width, empty, dtype=dtype, device=self.keys.device), empty)
        return self.col[name][0]

    def find(self, keys):
        at = torch.searchsorted(self.keys, keys).clamp(max=max(0, self.keys.shape[0] - 1))
        return at, (self.keys[at] == keys) if self.keys.shape[0] else torch.zeros_like(keys, dtype=torch.bool)


def _truncate(qo, qe, sample, voxel, max_range):
    d = (qe - qo).double()
    length = torch.sqrt(d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] + d[:, 2] * d[:, 2])
    rmax = max_range * (float(U) / voxel)
    far = length > rmax
    cut = qo + torch.round(d * (rmax / length)[:, None]).long()
    return torch.where(far[:, None], cut, qe), sample & ~far


def _integrate(tab, o, e, flags, case):
    """One call into `tab`: occupancy, NDT moments and voxel means."""
    voxel, names = case["voxel"], case["layers"].split("+")
    qo, qe = _quantise(o, voxel).expand(e.shape[0], 3), _quantise(e, voxel)
    qe, sample = _truncate(qo, qe, (flags & 1) == 0, voxel, case["range"])
    vox, ray, last = _walk(qo, qe)
    keys = _pack(vox.long())
    hit = last & sample[ray]
    mk, mc = torch.unique(keys[~hit], return_counts=True)
    ends = _pack(qe >> FRAC)[sample]
    hk, hc = torch.unique(ends, return_counts=True)
    tab.add(torch.cat([mk, hk]))
    l = tab.column("l", float("nan"), torch.float64)
    at, _ = tab.find(mk)
    l[at] = (torch.nan_to_num(l[at], nan=0.0) + mc.double() * W.MISS).clamp(min=-2.0)
    at, _ = tab.find(hk)
    l[at] = (torch.nan_to_num(l[at], nan=0.0) + hc.double() * W.HIT).clamp(max=3.5)
    p = (qe & (U - 1))[sample]
    at, _ = tab.find(ends)
    if "ndt" in names:
        x, y, z = p[:, 0], p[:, 1], p[:, 2]
        mom = torch.stack([torch.ones_like(x), x, y, z, x * x, x * y, x * z, y * y, y * z, z * z], 1)
        tab.column("mom", 0, torch.long, (10,)).index_add_(0, at, mom)
    if "mean" in names:
        mean = tab.column("mean", 0, torch.long, (4,))  # count, then x y z in 1/1024 voxel
        s = torch.zeros((tab.keys.shape[0], 4), dtype=torch.long, device=p.device)
        s.index_add_(0, at, torch.cat([torch.ones_like(p[:, :1]), p >> (FRAC - 10)], 1))
        has = s[:, 0] > 0
        n0, c = mean[has, 0], s[has, 0]
        nt = n0 + c
        mean[has, 1:] = (mean[has, 1:] * n0[:, None] + s[has, 1:] + (nt // 2)[:, None]) // nt[:, None]
        mean[has, 0] = nt


def _ndt_of(mom, vox, voxel):
    """(count, mean xyz, packed covariance) of moment sums, 64-bit."""
    n = mom[:, 0].double()
    has = n > 0
    nn = torch.where(has, n, torch.ones_like(n))
    cell = voxel / U
    s = mom[:, 1:4].double() / nn[:, None]
    mean = (vox.double() * U + s) * cell
    pa, pb = [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]
    num = mom[:, :1] * mom[:, 4:10] - mom[:, [1 + k for k in pa]] * mom[:, [1 + k for k in pb]]
    cov = num.double() / (nn * nn)[:, None] * cell * cell
    out = torch.cat([n[:, None], mean, cov], 1)
    return torch.where(has[:, None], out, torch.zeros_like(out))


def _lookup(tab, points, case):
    vox = _quantise(points, case["voxel"]) >> FRAC
    at, ok = tab.find(_pack(vox))
    names = case["layers"].split("+")
    l = tab.column("l", float("nan"), torch.float64)[at]
    out = dict(occupancy=torch.where(ok, l, torch.full_like(l, float("nan"))), known=None)
    if "ndt" in names:
        mom = torch.where(ok[:, None], tab.column("mom", 0, torch.long, (10,))[at], 0)
        out["ndt"] = _ndt_of(mom, vox, case["voxel"])
    if "counts" in names:
        out["counts"] = None
    if "decay" in names:
        out["path_sum"] = None
    if "mean" in names:
        m = torch.where(ok[:, None], tab.column("mean", 0, torch.long, (4,))[at], 0)
        pos = (vox.double() + (m[:, 1:].double() + 0.5) / 1024.0) * case["voxel"]
        pos = torch.where((m[:, :1] > 0), pos, torch.full_like(pos, float("nan")))
        out["mean"] = torch.cat([pos, m[:, :1].double()], 1)
    if "tsdf" in names:
        d = tab.column("D", 0.0, torch.float64)[at]
        w = tab.column("W", 0.0, torch.float64)[at]
        out["tsdf"] = torch.where(ok[:, None], torch.stack([d, w], 1), torch.zeros((1, 2), dtype=torch.float64, device=d.device))
    return out


def _depth_world(depth, K, pose, z_min=0.3, z_max=6.0):
    """World end points (float32), validity and R p~ of a depth frame's pixels."""
    h, w = depth.shape
    dev = depth.device
    px = ((torch.arange(w, dtype=torch.float64, device=dev) - K[2]) / K[0]).expand(h, w).reshape(-1)
    py = ((torch.arange(h, dtype=torch.float64, device=dev) - K[3]) / K[1])[:, None].expand(h, w).reshape(-1)
    z = depth.double().reshape(-1)
    valid = (z > z_min) & (z <= z_max)
    zz = torch.where(valid, z, torch.full_like(z, z_max))
    P = torch.from_numpy(pose).to(dev)
    x, y = px * zz, py * zz
    e = torch.stack([((P[k, 0] * x + P[k, 1] * y) + P[k, 2] * zz) + P[k, 3] for k in range(3)], 1).float()
    return e, valid, torch.stack([px, py, torch.ones_like(px)], 1) @ P[:, :3].T, P[:, 3].float()


def _band(e, valid, o, case):
    """The TSDF band of a frame: (voxels, ray of each, signed distance before
    the clamp, direction, length in metres, e - c)."""
    voxel, p = case["voxel"], W.tsdf_params()
    scale = float(U) / voxel
    qo, qe = _quantise(o[None], voxel).expand(e.shape[0], 3), _quantise(e, voxel)
    d = (qe - qo).double()
    length = torch.sqrt(d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1] + d[:, 2] * d[:, 2])
    use = torch.nonzero(valid & (length > p["min_range"] * scale) & (length <= p["max_range"] * scale))[:, 0]
    qo, qe, d, length = qo[use], qe[use], d[use], length[use]
    tau = case["trunc"] * scale
    a = qo + torch.round(d * ((length - tau).clamp(min=0.0) / length)[:, None]).long()
    b = qo + torch.round(d * ((length + tau) / length)[:, None]).long()
    vox, ray, _ = _walk(a, b)
    u = d / length[:, None]
    r = (qe[ray] - (vox.long() * U + U // 2)).double() * (voxel / U)
    return vox.long(), use[ray], (r * u[ray]).sum(1), u[ray], (length * voxel / U)[ray], r


def _integrate_depth(tab, frame, case):
    e, valid, _, o = _depth_world(*frame)
    vox, ray, s, u, length, r = _band(e, valid, o, case)
    keys = _pack(vox)
    tab.add(torch.unique(keys))
    at, _ = tab.find(keys)
    D, Wt = tab.column("D", 0.0, torch.float64), tab.column("W", 0.0, torch.float64)
    S = torch.zeros_like(D).index_add_(0, at, s.clamp(-case["trunc"], case["trunc"]))
    C = torch.zeros_like(D).index_add_(0, at, torch.ones_like(s))
    has = C > 0
    D[has] = (Wt[has] * D[has] + S[has]) / (Wt[has] + C[has])
    Wt[has] = (Wt[has] + C[has]).clamp(max=float(1 << 20))
    return e, ray, at, s, u, length, r, o


def _exact_tsdf_grad(case, seed):
    depth, K, pose, pts, grad = _grad_inputs(case, seed)
    tab = _Table(depth.device)
    e, ray, at, s, u, length, r, o = _integrate_depth(tab, (depth, K, pose), case)
    q, ok = tab.find(_pack(_quantise(pts, case["voxel"]) >> FRAC))
    D = torch.where(ok, tab.column("D", 0.0, torch.float64)[q], 0.0)
    G = torch.zeros(tab.keys.shape[0], dtype=torch.float64, device=depth.device).index_add_(0, q, torch.where(ok, grad.double(), 0.0))
    w = torch.where(s.abs() < case["trunc"], (G / tab.column("W", 0.0, torch.float64).clamp(min=1.0))[at], 0.0)
    n = depth.numel()
    zero = torch.zeros(n, 3, dtype=torch.float64, device=depth.device)
    ge = zero.clone().index_add_(0, ray, w[:, None] * (u + (r - s[:, None] * u) / length[:, None]))
    go = zero.clone().index_add_(0, ray, -w[:, None] * (r - s[:, None] * u) / length[:, None])
    _, _, Rp, _ = _depth_world(depth, K, pose)
    E, O = e.double(), o.double().expand(n, 3)
    twist = torch.cat([(ge + go).sum(0), (torch.linalg.cross(E, ge) + torch.linalg.cross(O, go)).sum(0)])
    return dict(distance=D, grad_depth=(ge * Rp).sum(1).reshape(depth.shape), grad_twist=twist.cpu())


def _exact_ndt_grad(case, seed):
    ray, pose, pts, gmean, gcov = _grad_inputs(case, seed)
    dev, voxel = pts.device, case["voxel"]
    P = torch.from_numpy(pose).to(dev)

    def move(x):
        x = x.double()
        return torch.stack([((P[k, 0] * x[:, 0] + P[k, 1] * x[:, 1]) + P[k, 2] * x[:, 2]) + P[k, 3] for k in range(3)], 1).float()

    o, e = move(ray.origins), move(ray.endpoints)
    c = dict(case, layers="occ+ndt")
    tab = _Table(dev)
    _integrate(tab, o, e, ray.flags, c)
    stats = _lookup(tab, pts, c)["ndt"]
    q, ok = tab.find(_pack(_quantise(pts, voxel) >> FRAC))
    g = torch.zeros((tab.keys.shape[0], 9), dtype=torch.float64, device=dev)
    g.index_add_(0, q, torch.where(ok[:, None], torch.cat([gmean, gcov], 1).double(), 0.0))
    qo, qe = _quantise(o, voxel).expand(e.shape[0], 3), _quantise(e, voxel)
    _, sample = _truncate(qo, qe, (ray.flags & 1) == 0, voxel, case["range"])
    at, found = tab.find(_pack(qe >> FRAC))
    mom = tab.column("mom", 0, torch.long, (10,))[at].double()
    n = mom[:, :1].clamp(min=1.0)
    d = ((qe & (U - 1)).double() - mom[:, 1:4] / n) * (voxel / U)
    w = g[at]
    H = torch.stack([2 * w[:, 3], w[:, 4], w[:, 5], w[:, 4], 2 * w[:, 6], w[:, 7], w[:, 5], w[:, 7], 2 * w[:, 8]], 1).reshape(-1, 3, 3)
    gp = (w[:, :3] + (H @ d[:, :, None])[:, :, 0]) / n
    gp = torch.where((sample & found)[:, None], gp, 0.0)
    twist = torch.cat([gp.sum(0), torch.linalg.cross(e.double(), gp).sum(0)])
    return dict(mean=stats[:, 1:4], cov=stats[:, 4:10], grad_endpoints=gp @ P[:, :3], grad_twist=twist.cpu())


def exact(case, seed):
    kind, dev = case["kind"], _dev()
    if kind == "scan":
        ring = [_scan(case, seed, k) for k in range(case["ring"])]
        tab = _Table(dev)
        for r in ring[1:] + ring[:1]:
            _integrate(tab, r.origins, r.endpoints, r.flags, case)
        return _lookup(tab, _points(case, ring[0]), case)
    if kind == "build":
        scans = _outdoor(case, seed)
        tab = _Table(dev)
        for r in scans:
            _integrate(tab, r.origins, r.endpoints, r.flags, case)
        return _lookup(tab, _points(case, scans[-1]), case)
    if kind == "depth":
        if "occ" in case["layers"].split("+"):
            return None
        frames = [_depth(case, seed, k) for k in range(case["ring"])]
        tab = _Table(dev)
        for f in frames[1:] + frames[:1]:
            _integrate_depth(tab, f, case)
        out = _lookup(tab, _surface_points(*frames[0], case["stride"]), dict(case))
        out["occupancy"] = torch.full_like(out["occupancy"], float("nan"))
        return out
    if kind == "tsdf_grad":
        return _exact_tsdf_grad(case, seed)
    if kind == "ndt_grad":
        return _exact_ndt_grad(case, seed)
    if kind == "fleet":
        occ = []
        for p, r, pts in _fleet(case, seed):
            c = dict(case, voxel=p["voxel_size"], range=p["max_range"], layers="occ")
            tab = _Table(dev)
            _integrate(tab, r.origins, r.endpoints, r.flags, c)
            occ.append(_lookup(tab, pts, c)["occupancy"])
        return dict(occupancy=occ, known=[None] * len(occ))
    if kind == "publish":
        ray = _publish_scan(case, seed)
        tab = _Table(dev)
        one = torch.ones(1, dtype=torch.uint8, device=dev)
        regions = []
        for p in _first_rays(case):
            _integrate(tab, p.to(dev), p.to(dev), one, case)
            regions.append(((_quantise(p, case["voxel"])[0]) >> FRAC) >> 5)
        _integrate(tab, ray.origins, ray.endpoints, ray.flags, case)
        lin = torch.arange(32768, device=dev)
        local = torch.stack([lin & 31, (lin >> 5) & 31, lin >> 10], 1)
        vox = torch.stack(regions).to(dev)[:, None, :] * 32 + local[None]
        at, ok = tab.find(_pack(vox.reshape(-1, 3)))
        l = tab.column("l", float("nan"), torch.float64)[at]
        around = _lookup(tab, _points(case, ray), case)
        dense = torch.where(ok, l, torch.full_like(l, float("nan"))).reshape(len(regions), 32768)
        out = dict(keys=None, occupancy=dense)
        for name in ("counts", "ndt"):
            if name in case["layers"].split("+"):
                out[name] = None
        return dict(map=out, around=around)
    return None
