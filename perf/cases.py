"""The work a user of the renderer has it do, as cases that can be timed and checked.

Scenes are driving-scene-shaped voxel sets (a ground slab of 0.2 m voxels, car-sized shells and
poles of 0.1 m voxels) or a small cube of scattered voxels, drawn on the GPU from a seed; sensors
stand on the scene's road at seeded poses.  `exact` states every output in 64 bits: a plain
cell-by-cell walk of the level-0 grid, a sort of each ray's hits by entry, and the compositing
sums and their adjoint written out with torch.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2507_18713_gb300 as salf

DEV = "cuda"
C0 = 0.5 / math.sqrt(math.pi)            # SH band 0
C1 = math.sqrt(3.0) / (2.0 * math.sqrt(math.pi))  # SH band 1
T_MIN = 1e-4                              # the renderer's default early-termination bound


# ------------------------------------------------------------------ the cases

def listed():
    cam = dict(sensor="pinhole", hfov=60.0)
    return [
        # an interactive preview of a small captured object: launch and latency
        dict(name="preview_128x96", path="render", **cam, w=128, h=96, scene="scatter", n=4096,
             dtype="f32", mode="exp"),
        # the front camera of a simulated drive, one frame
        dict(name="camera_1080p", path="render", **cam, w=1920, h=1080, scene="driving",
             n=2_000_000, dtype="f32", mode="exp"),
        # one LiDAR sweep with motion: range and intensity
        dict(name="lidar_128x2048", path="render", sensor="lidar", w=2048, h=128,
             scene="driving", n=2_000_000, dtype="f32", mode="exp"),
        # a wide surround camera
        dict(name="fisheye_1080p", path="render", sensor="fisheye", hfov=190.0, w=1920, h=1080,
             scene="driving", n=2_000_000, dtype="f32", mode="exp"),
        # every sensor of a vehicle asks the resident scene's server for its frame at once:
        # 8 cameras, 4 fisheyes, 2 panoramas, 4 large and 2 small LiDARs
        dict(name="serve_20_sensors", path="serve", cameras=8, fisheyes=4, panoramas=2, lidars=4,
             small_lidars=2, scale=1.0, scene="driving", n=4_000_000, dtype="bf16", mode="exp"),
        # one optimisation step of a scene: 8 views forward, image loss, adjoint
        dict(name="train_8x960x640", path="train", **cam, w=960, h=640, views=8, scene="driving",
             n=1_000_000, dtype="bf16", mode="exp"),
        # fitting an SDF scene to one LiDAR sweep: range, opacity and intensity gradients
        dict(name="lidar_fit_64x1024", path="lidar_fit", sensor="lidar", w=1024, h=64,
             scene="driving", n=500_000, dtype="f32", mode="sdf"),
        # the smoothness term of the same optimisation, over all neighbouring voxels
        dict(name="regularise_1M", path="regularise", scene="driving", n=1_000_000, dtype="f32",
             mode="sdf"),
        # a densify / prune step: new voxel list and the scene rebuilt from it
        dict(name="densify_rebuild_1M", path="densify", scene="driving", n=1_000_000,
             dtype="bf16", mode="exp"),
        # a 4K frame by tile rasterisation
        dict(name="raster_4k", path="raster", **cam, w=3840, h=2160, scene="driving", n=2_000_000,
             dtype="f32", mode="exp"),
        # the front camera with moving traffic
        dict(name="traffic_camera_1080p", path="actors", **cam, w=1920, h=1080, actors=24,
             scene="driving", n=2_000_000, dtype="f32", mode="exp"),
        # reflections off a rendered frame: spawn and trace
        dict(name="reflect_1080p", path="reflect", **cam, w=1920, h=1080, scene="driving",
             n=2_000_000, dtype="f32", mode="exp"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes, sensors, storage types and field modes over the listed range."""
    path = rng.choice(["render", "render", "render", "serve", "train", "lidar_fit", "regularise",
                       "densify", "raster", "raster", "actors", "reflect"])
    c = dict(path=path, scene="driving", dtype=rng.choice(["f32", "bf16"]),
             mode=rng.choice(["exp", "exp", "sdf"]))
    if path == "render":
        c["sensor"] = rng.choice(["pinhole", "pinhole", "fisheye", "pano", "lidar"])
        if rng.random() < 0.25:
            c.update(scene="scatter", n=_log_int(rng, 1500, 60_000))
        else:
            c["n"] = _log_int(rng, 100_000, 4_000_000)
    elif path == "serve":
        c.update(cameras=rng.randint(1, 6), fisheyes=rng.randint(0, 3),
                 panoramas=rng.randint(0, 1), lidars=rng.randint(1, 4),
                 small_lidars=rng.randint(0, 2), scale=round(rng.uniform(0.3, 1.0), 2),
                 n=_log_int(rng, 500_000, 4_000_000))
        return c
    elif path in ("regularise", "densify"):
        c["n"] = _log_int(rng, 30_000, 2_000_000)
        return c
    elif path == "lidar_fit":
        c["sensor"] = "lidar"
        c["n"] = _log_int(rng, 100_000, 1_500_000)
    else:
        c["sensor"] = "pinhole"
        c["n"] = _log_int(rng, 200_000, 2_500_000)
    if c["sensor"] == "lidar":
        c.update(w=_log_int(rng, 400, 2400), h=_log_int(rng, 16, 128))
    elif c["sensor"] == "pano":
        w = _log_int(rng, 512, 4096)
        c.update(w=w, h=max(64, w // 4 + rng.randint(-9, 9)))
    else:
        lo, hi = {"train": (200, 960), "raster": (480, 3840), "reflect": (320, 1920)}.get(
            path, (160, 2560))
        w = _log_int(rng, lo, hi)
        c.update(w=w, h=max(16, int(w * rng.uniform(0.5, 0.75))),
                 hfov=round(rng.uniform(170.0, 200.0) if c["sensor"] == "fisheye"
                            else rng.uniform(40.0, 100.0), 1))
    if path == "train":
        c["views"] = rng.randint(1, 8)
    if path == "actors":
        c["actors"] = rng.randint(3, 24)
    return c


# ------------------------------------------------------------------ scenes

def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1009 + salt)


def _u(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)


def _records(g, n, mode):
    """Voxel records: densities log-normal around 1 per metre (or an SDF through the voxel),
    colours spread over (0, 1), small slopes and view dependence."""
    def nrm(s, *shape):
        return s * torch.randn(shape, generator=g, device=DEV)
    p = torch.zeros((n, 32), device=DEV)
    if mode == "exp":
        p[:, 0:3] = nrm(0.25, n, 3)
        p[:, 3] = nrm(1.0, n)
    else:
        p[:, 0:4] = nrm(0.5, n, 4)
    p[:, 4:13] = nrm(0.1, n, 9)
    p[:, 13:25] = nrm(0.1, n, 12)
    p[:, [13, 17, 21]] = _u(g, -12.0, 12.0, n, 3).float()
    p[:, 25] = nrm(1.0, n).exp()
    p[:, 26] = _u(g, 0.05, 0.5, n).float()
    p[:, 27:30] = nrm(0.1, n, 3)
    p[:, 30] = _u(g, -4.0, 4.0, n).float()
    return p


def _box_shell(nx, ny, nz):
    i, j, k = torch.meshgrid(*(torch.arange(m, device=DEV) for m in (nx, ny, nz)), indexing="ij")
    on = (i == 0) | (i == nx - 1) | (j == 0) | (j == ny - 1) | (k == 0) | (k == nz - 1)
    return torch.stack([i[on], j[on], k[on]], 1)


def _driving(g, n):
    """Level and cell of n disjoint voxels: half of them ground, the rest parked cars (about
    3,450 voxels each) and some poles, which keep clear of the road |y| < 4 m."""
    layers = 2 if n > 2_500_000 else 1
    side = min(1000, int(math.sqrt(0.5 * n / layers)))
    a = torch.arange(side, device=DEV) + 512 - side // 2
    gi, gj, gk = torch.meshgrid(a, a, torch.arange(layers, device=DEV), indexing="ij")
    ground = torch.stack([gi.reshape(-1), gj.reshape(-1), gk.reshape(-1)], 1)[:n]
    rest = n - ground.shape[0]
    half = 0.1 * side - 3.0

    def spots(m):
        x, y = _u(g, -half, half, m), _u(g, 7.0, max(half, 10.0), m)
        return x, torch.where(_u(g, 0.0, 1.0, m) < 0.5, -y, y)

    # cars, in 8 sizes
    cars = max(1, int(0.95 * rest / 3450))
    parts = []
    for q in range(8):
        m = (cars + 7 - q) // 8
        if m == 0:
            continue
        s = _u(g, 0.0, 1.0, 4).tolist()
        nx, ny, nz = 35 + int(15 * s[0]), 17 + int(5 * s[1]), 14 + int(5 * s[2])
        shell = _box_shell(*((ny, nx, nz) if s[3] < 0.5 else (nx, ny, nz)))
        x, y = spots(m)
        o = torch.stack([((x + 102.4) / 0.1).long() - 20, ((y + 102.4) / 0.1).long() - 20,
                         torch.full((m,), 2 * layers, device=DEV)], 1)
        parts.append((o[:, None, :] + shell[None]).reshape(-1, 3))
    # poles 3-8 m high, more than are needed
    m = int(0.4 * rest / 55) + 200
    x, y = spots(m)
    h = _u(g, 30.0, 80.0, m).long()
    k = torch.arange(80, device=DEV)
    keep = k[None] < h[:, None]
    base = torch.stack([((x + 102.4) / 0.1).long(), ((y + 102.4) / 0.1).long(),
                        torch.full((m,), 2 * layers, device=DEV)], 1)
    poles = base[:, None, :].repeat(1, 80, 1)
    poles[..., 2] += k
    parts.append(poles[keep])
    fine = torch.cat(parts)
    # each cell once, the first that names it
    key = (fine[:, 0] * 2048 + fine[:, 1]) * 256 + fine[:, 2]
    _, inv = torch.unique(key, return_inverse=True)
    at = torch.arange(fine.shape[0], device=DEV)
    first = torch.full((int(inv.max()) + 1,), fine.shape[0], device=DEV).scatter_reduce(
        0, inv, at, "amin")
    fine = fine[first.sort().values][:rest]
    level = torch.cat([torch.zeros(ground.shape[0], device=DEV),
                       torch.ones(fine.shape[0], device=DEV)]).to(torch.uint8)
    return level, torch.cat([ground, fine]).to(torch.int32)


def _voxels(case, seed):
    g = _gen(seed, 1)
    n = case["n"]
    if case["scene"] == "scatter":
        d = 64
        cell = torch.randperm(d ** 3, generator=g, device=DEV)[:n]
        ijk = torch.stack([cell % d, cell // d % d, cell // (d * d)], 1).to(torch.int32)
        level = torch.zeros(ijk.shape[0], dtype=torch.uint8, device=DEV)
        return salf.VoxelSet((0.0, 0.0, 0.0), 0.1, (d, d, d), 0, level, ijk,
                             _records(g, ijk.shape[0], case["mode"]), case["mode"])
    level, ijk = _driving(g, n)
    return salf.VoxelSet((-102.4, -102.4, 0.0), 0.2, (1024, 1024, 128), 1, level, ijk,
                         _records(g, ijk.shape[0], case["mode"]), case["mode"])


def _car(g, seed, mode):
    """A car in its own frame: a floor of 0.2 m voxels under a shell of 0.1 m voxels."""
    s = _u(g, 0.0, 1.0, 3).tolist()
    nx, ny, nz = 20 + int(4 * s[0]), 9 + int(2 * s[1]), 7 + int(2 * s[2])
    fi, fj = torch.meshgrid(torch.arange(nx, device=DEV), torch.arange(ny, device=DEV),
                            indexing="ij")
    floor = torch.stack([fi.reshape(-1), fj.reshape(-1), torch.zeros_like(fi.reshape(-1))], 1)
    shell = _box_shell(2 * nx, 2 * ny, 2 * nz)
    shell = shell[shell[:, 2] >= 2]
    level = torch.cat([torch.zeros(floor.shape[0], device=DEV),
                       torch.ones(shell.shape[0], device=DEV)]).to(torch.uint8)
    ijk = torch.cat([floor, shell]).to(torch.int32)
    return salf.VoxelSet((-0.1 * nx, -0.1 * ny, 0.0), 0.2, (nx, ny, nz), 1, level, ijk,
                         _records(g, ijk.shape[0], mode), mode)


# ------------------------------------------------------------------ sensors

def _yaw(a):
    c, s = math.cos(a), math.sin(a)
    return np.array([[c, -s, 0.0], [s, c, 0.0], [0.0, 0.0, 1.0]])


def _pose(rot, pos):
    return np.concatenate([rot, np.asarray(pos, float).reshape(3, 1)], 1)


def _camera(pos, yaw):
    c, s = math.cos(yaw), math.sin(yaw)
    return _pose(np.array([[s, 0.0, c], [-c, 0.0, s], [0.0, -1.0, 0.0]]), pos)


def _sensor(kind, w, h, pose0, pose1=None, hfov=60.0):
    s = dict(kind=kind, width=w, height=h, fx=0.0, fy=0.0, cx=0.0, cy=0.0, fov=0.0, elev_min=0.0,
             elev_max=0.0, pose0=pose0, pose1=pose0 if pose1 is None else pose1, t0=0.0, t1=0.0,
             rolling_shutter=False, t_near=0.0, t_far=0.0, rays=None)
    if kind == "pinhole":
        f = 0.5 * w / math.tan(0.5 * math.radians(hfov))
        s.update(fx=f, fy=f, cx=0.5 * w, cy=0.5 * h)
    elif kind == "fisheye":
        s.update(fx=w / math.radians(hfov), fy=w / math.radians(hfov), cx=0.5 * w, cy=0.5 * h,
                 fov=math.radians(hfov))
    elif kind == "pano":
        s.update(elev_min=-math.pi * h / w, elev_max=math.pi * h / w)
    else:
        s.update(elev_min=math.radians(-25.0), elev_max=math.radians(15.0), t1=0.1,
                 rolling_shutter=True)
    return s


def _place(kind, w, h, r, hfov=60.0, scene="driving", yaw=None, spread=3.0):
    """A sensor at a seeded pose: on the road, or before the cube of scattered voxels."""
    if scene == "scatter":
        p = [3.2 + 0.3 * r.uniform(-1, 1), -5.0 + r.uniform(-1, 1), 3.2 + 0.3 * r.uniform(-1, 1)]
        a = math.pi / 2 + r.uniform(-0.05, 0.05)
    else:
        p = [r.uniform(-spread, spread), r.uniform(-1.5, 1.5), 1.7 + r.uniform(-0.15, 0.15)]
        a = r.uniform(-0.2, 0.2) if yaw is None else yaw + r.uniform(-0.05, 0.05)
    if kind == "lidar":
        p[2] += 0.2
        p1 = [p[0] + r.uniform(0.0, 1.2), p[1], p[2]]
        return _sensor(kind, w, h, _pose(_yaw(a), p), _pose(_yaw(a + 0.02), p1))
    return _sensor(kind, w, h, _camera(p, a), hfov=hfov)


def _wants(kind):
    if kind == "lidar":
        return dict(want_intensity=True, outputs=("depth", "opacity", "intensity"))
    return dict(want_intensity=False, outputs=("rgb", "depth", "opacity"))


def _sensors(case, seed):
    r = np.random.default_rng(int(seed) + 77)
    if case["path"] == "train":
        return [_place("pinhole", case["w"], case["h"], r, case["hfov"],
                       yaw=k * 2.0 * math.pi / case["views"]) for k in range(case["views"])]
    if case["path"] == "serve":
        s = case["scale"]
        kinds = ([("pinhole", 1920, 1080, 60.0)] * case["cameras"]
                 + [("fisheye", 1280, 960, 190.0)] * case["fisheyes"]
                 + [("pano", 4096, 1024, 0.0)] * case["panoramas"]
                 + [("lidar", 2048, 128, 0.0)] * case["lidars"]
                 + [("lidar", 1024, 64, 0.0)] * case["small_lidars"])
        return [_place(k, int(w * s), int(h * s), r, f, yaw=r.uniform(0.0, 2.0 * math.pi),
                       spread=20.0) for k, w, h, f in kinds]
    return [_place(case["sensor"], case["w"], case["h"], r, case.get("hfov", 60.0), case["scene"])]


def _traffic(case, seed):
    """Cars in two lanes ahead of and behind the camera: (voxels, pose at t0, pose at t1)."""
    g = _gen(seed, 5)
    r = np.random.default_rng(int(seed) + 5)
    slots = [(s * (10.0 + 8.0 * k) + r.uniform(0.0, 1.5) * s, y) for k in range(6)
             for s in (1.0, -1.0) for y in (-2.0, 2.0)]
    out = []
    for q in sorted(r.choice(len(slots), case["actors"], replace=False).tolist()):
        x, y = slots[q]
        a = (0.0 if y < 0 else math.pi) + r.uniform(-0.05, 0.05)
        step = 0.1 * r.uniform(0.0, 12.0)
        p0 = _pose(_yaw(a), (x, y, 0.2))
        p1 = _pose(_yaw(a + 0.1 * r.uniform(-0.3, 0.3)),
                   (x + step * math.cos(a), y + step * math.sin(a), 0.2))
        out.append((_car(g, seed, case["mode"]), p0, p1))
    return out


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    path = case["path"]
    vox = _voxels(case, seed)
    st = dict(case=case, vox=vox)
    if path != "densify":
        st["scene"] = salf.Scene(vox, dtype=case["dtype"])
    g = _gen(seed, 3)
    if path == "regularise":
        return st
    if path == "densify":
        n = vox.params.shape[0]
        st["scene"] = salf.Scene(vox, dtype=case["dtype"])
        # a training pass's gradients: a twentieth of the voxels (ground, as only level 0 can be
        # split) stand out by their colour slopes; one in fifty is nearly transparent
        grads = torch.randn((n, 32), generator=g, device=DEV)
        size = 0.8 * torch.rand(n, generator=g, device=DEV)
        pick = torch.randperm(int((vox.level == 0).sum()), generator=g, device=DEV)
        size[pick[:n // 20]] += 1.5
        st["grads"] = grads * (size / grads[:, 4:13].abs().sum(1))[:, None]
        st["threshold"] = 1.0
        alpha = 0.05 + 0.9 * torch.rand(n, generator=g, device=DEV)
        alpha[pick[n // 20:n // 20 + n // 50]] = 1e-4
        st["max_alpha"] = alpha
        return st
    st["sensors"] = _sensors(case, seed)
    sen = st["sensors"][0]
    if path == "serve":
        st["server"] = salf.Server(st["scene"], 8 << 30, 4)
    elif path == "train":
        st["params"] = vox.params.clone().requires_grad_(True)
        R = case["w"] * case["h"]
        st["targets"] = [torch.rand((R, 3), generator=g, device=DEV) for _ in st["sensors"]]
    elif path == "lidar_fit":
        R = case["w"] * case["h"]
        st["loss_grads"] = [torch.randn(R, generator=g, device=DEV) / R for _ in range(3)]
    elif path == "actors":
        st["cars"] = [(salf.Scene(v, dtype=case["dtype"]), p0, p1, (k + 1) << 22)
                      for k, (v, p0, p1) in enumerate(_traffic(case, seed))]
    elif path == "reflect":
        first = st["scene"].render(sen)
        st["depth"], st["opacity"] = first["depth"], first["opacity"]
    return st


def run(st):
    case, scene, path = st["case"], st["scene"], st["case"]["path"]
    if path == "regularise":
        loss, grads = scene.reg_loss(st["vox"].params, 0.01, 0.02, 0.03)
        return dict(loss=loss, grads=grads)
    if path == "densify":
        new, counts = scene.refine(st["vox"].params, st["grads"], st["max_alpha"],
                                   st["threshold"])
        st["rebuilt"] = salf.Scene(new, dtype=case["dtype"])
        info = st["rebuilt"].info()
        records = st["rebuilt"].params_view()  # the scene's own memory: a copy outlives it
        if case["dtype"] == "bf16":
            records = records.view(torch.int16)
        return dict(level=new.level, ijk=new.ijk, params=new.params, counts=counts,
                    records=records.clone(), cells=info["n_level0_cells"], nodes=info["n_nodes"])
    sensors = st["sensors"]
    if path == "serve":
        # one time step: the requests start together; the results are copied out, and the
        # server gets its memory back once the copies are done
        server = st["server"]
        server.hold(True)
        tickets = [server.submit(s, want_intensity=s["kind"] == "lidar") for s in sensors]
        server.hold(False)
        outs = []
        for t, s in zip(tickets, sensors):
            got = server.fetch(t)
            outs.append([got[k] for k in _wants(s["kind"])["outputs"]])
        torch.cuda.current_stream().synchronize()
        for t in tickets:
            server.release(t)
        return outs
    if path == "train":
        flat = salf.RenderBatchFn.apply(st["params"], scene, sensors)
        loss = sum(torch.nn.functional.mse_loss(flat[3 * k], t)
                   for k, t in enumerate(st["targets"]))
        grads, = torch.autograd.grad(loss, st["params"])
        return dict(loss=loss.detach(), grads=grads, rgb=[t.detach() for t in flat[0::3]])
    sen = sensors[0]
    if path == "render":
        out = scene.render(sen, **_wants(sen["kind"]))
    elif path == "lidar_fit":
        out = scene.render(sen, saved=True, **_wants("lidar"))
        d, o, i = st["loss_grads"]
        out["grads"] = scene.backward(sen, out["saved"], d_depth=d, d_opacity=o, d_intensity=i,
                                      want_intensity=True)
        out.pop("saved")
    elif path == "raster":
        out = scene.render_raster(sen)
    elif path == "actors":
        out = scene.render_actors(sen, st["cars"])
    else:
        rays = scene.secondary_rays(sen, st["depth"], st["opacity"], kind="reflect")
        out = dict(scene.render(salf.rays_sensor(rays)), rays=rays)
    out.pop("_keep", None)
    return out


# ------------------------------------------------------------------ work

def work(case):
    """Bytes and operations of one pass: every record that is seen and every input read once,
    every output written once; about 200 operations a ray (its set-up and its end) and 110 a
    voxel it crosses, of which the scenes here hold 6 a ray."""
    n, rec = case["n"], 100 if case["dtype"] == "f32" else 50
    path = case["path"]
    if path == "regularise":
        return dict(bytes=n * (16 + 24 + 2 * 24), flops=2.5 * n * 90)
    if path == "densify":
        m = 1.3 * n
        out = m * (13 + 128) + m * (128 if case["dtype"] == "f32" else 64)
        return dict(bytes=n * (13 + 128 + 36 + 4) + m * (13 + 128) + out, flops=m * 60)
    if path == "serve":
        s2 = case["scale"] ** 2
        rays = s2 * (1920 * 1080 * case["cameras"] + 1280 * 960 * case["fisheyes"]
                     + 4096 * 1024 * case["panoramas"] + 2048 * 128 * case["lidars"]
                     + 1024 * 64 * case["small_lidars"])
        return dict(bytes=n * rec + rays * 21, flops=rays * 860)
    rays = case["w"] * case["h"]
    hits = rays * 6.0
    seen = min(n * (case.get("hfov", 360.0) / 360.0 if case["sensor"] == "pinhole" else 1.0), hits)
    if path == "train":
        v = case["views"]
        seen = min(n, seen * v)
        return dict(bytes=n * (128 + 64 + 128) + 2 * seen * rec + seen * 100
                    + v * rays * (12 + 12 + 32 + 32 + 12), flops=v * rays * 860 * 3.5)
    if path == "lidar_fit":
        return dict(bytes=n * 128 + 2 * seen * 124 + seen * 124 + rays * (13 + 64 + 12),
                    flops=rays * 860 * 3.5)
    if path == "reflect":
        return dict(bytes=rays * (8 + 64 + 21) + 2 * seen * rec, flops=rays * 900)
    return dict(bytes=rays * 21 + seen * rec, flops=rays * 860)


# ------------------------------------------------------------------ the same in 64 bits

class _Grid:
    """A voxel set as a dense table of its level-0 cells: the voxel, or 8 children."""

    def __init__(self, vox, dtype):
        self.s0, self.mode = vox.s0, vox.mode
        self.origin = torch.tensor(vox.origin, device=DEV, dtype=torch.float64)
        p = vox.params
        self.params = (p.bfloat16() if dtype == "bf16" else p).double()
        self.dims = tuple(vox.dims)
        lev, ijk = vox.level.long(), vox.ijk.long()
        cell = ijk >> lev[:, None]
        flat = (cell[:, 2] * self.dims[1] + cell[:, 1]) * self.dims[0] + cell[:, 0]
        ids = torch.arange(lev.shape[0], device=DEV)
        self.table = torch.full((self.dims[0] * self.dims[1] * self.dims[2],), -1, device=DEV,
                                dtype=torch.int32)
        whole = lev == 0
        self.table[flat[whole]] = ids[whole].int()
        split, inv = torch.unique(flat[~whole], return_inverse=True)
        self.kids = torch.full((max(1, split.shape[0]), 8), -1, device=DEV, dtype=torch.long)
        c = ijk[~whole] & 1
        self.kids[inv, c[:, 0] | c[:, 1] << 1 | c[:, 2] << 2] = ids[~whole]
        self.table[split] = (-2 - torch.arange(split.shape[0], device=DEV)).int()
        self.level, self.ijk = lev, ijk
        self.lo = cell.min(0).values
        self.hi = cell.max(0).values + 1

    def box(self, v):
        edge = self.s0 / (1 << self.level[v]).double()
        lo = self.ijk[v].double() * edge[:, None]
        return lo, edge

    def hits(self, o, d, tn, tf):
        """(ray, voxel, entry, exit) of every voxel that the rays cross, in no order; o is
        relative to the world, distances are along the unit direction d."""
        o = o - self.origin
        d = torch.where(d == 0, torch.full_like(d, 1e-300), d)
        inv = 1.0 / d
        a = (self.lo.double() * self.s0 - o) * inv
        b = (self.hi.double() * self.s0 - o) * inv
        t0 = torch.maximum(torch.minimum(a, b).amax(1), tn)
        t1 = torch.minimum(torch.maximum(a, b).amin(1), tf)
        ray = (t0 < t1).nonzero()[:, 0]
        og, dg, iv, t1 = o[ray] / self.s0, d[ray], inv[ray] * self.s0, t1[ray]
        c = torch.floor(og + dg / self.s0 * t0[ray][:, None]).long()
        c = torch.maximum(torch.minimum(c, self.hi - 1), self.lo)
        up = (dg > 0)
        step = torch.where(up, 1, -1)
        tmax = (c + up.long() - og) * iv
        dt = iv.abs()
        rays, cells = [], []
        turn = 0
        stride = torch.tensor([1, self.dims[0], self.dims[0] * self.dims[1]], device=DEV)
        while ray.numel():
            flat = (c * stride).sum(1)
            on = self.table[flat] != -1
            rays.append(ray[on])
            cells.append(flat[on])
            t, ax = tmax.min(1)
            one = torch.nn.functional.one_hot(ax, 3)
            c = c + step * one
            tmax = torch.where(one.bool(), tmax + dt, tmax)
            live = (t < t1) & ((c >= self.lo) & (c < self.hi)).all(1)
            # a ray that has left stays on the spot until the next sweep
            t1 = torch.where(live, t1, torch.full_like(t1, -1.0))
            c = torch.where(live[:, None], c, self.lo)
            turn += 1
            if turn % 4 == 0 or ray.numel() < 20_000:
                ray, og, iv, t1, c, tmax, dt, step = (
                    x[live] for x in (ray, og, iv, t1, c, tmax, dt, step))
            else:
                ray = torch.where(live, ray, -1)
        none = torch.zeros(0, dtype=torch.long, device=DEV)
        ray, e = torch.cat([none] + rays), self.table[torch.cat([none] + cells)].long()
        e, ray = e[ray >= 0], ray[ray >= 0]
        kid = self.kids[(-2 - e[e < -1])]
        ray = torch.cat([ray[e >= 0], ray[e < -1].repeat_interleave(8)])
        v = torch.cat([e[e >= 0], kid.reshape(-1)])
        ray, v = ray[v >= 0], v[v >= 0]
        lo, edge = self.box(v)
        a, b = (lo - o[ray]) * inv[ray], (lo + edge[:, None] - o[ray]) * inv[ray]
        tin = torch.maximum(torch.minimum(a, b).amax(1), tn[ray])
        tout = torch.minimum(torch.maximum(a, b).amin(1), tf[ray])
        on = tout > tin
        return ray[on], v[on], tin[on], tout[on]

    def field(self, o, d, ray, v, tin, tout, intensity=False):
        """Optical depth and field values of the hits at their segments' midpoints."""
        tm = 0.5 * (tin + tout)
        lo, edge = self.box(v)
        x = (o[ray] - self.origin + tm[:, None] * d[ray] - lo) / (0.5 * edge[:, None]) - 1.0
        p = self.params[v]
        dd = d[ray]
        gam = torch.stack([torch.full_like(tm, C0), C1 * dd[:, 1], C1 * dd[:, 2], C1 * dd[:, 0]], 1)
        lin = (p[:, 0:3] * x).sum(1) + p[:, 3]
        if self.mode == "exp":
            sig = lin.exp()
        else:
            sig = 0.5 * p[:, 25] * (1.0 + lin.sign() * (1.0 - torch.exp(-lin.abs() / p[:, 26])))
        z = (p[:, 4:13].view(-1, 3, 3) * x[:, None]).sum(2) + (
            p[:, 13:25].view(-1, 3, 4) * gam[:, None]).sum(2)
        q = [torch.sigmoid(z), tm[:, None]]
        if intensity:
            q.append(torch.sigmoid((p[:, 27:30] * x).sum(1) + p[:, 30])[:, None])
        return dict(ray=ray, v=v, tin=tin, len=tout - tin, sig=sig, lin=lin, x=x, gam=gam,
                    q=torch.cat(q, 1))


def _composite(h, R, q=None):
    """Front-to-back sums over the hits, sorted in place by ray and entry; stops each ray after
    the hit that takes its transmittance below the bound.  Returns per-ray sums of q and 1 - T,
    with the hits that count and the transmittance before and after each."""
    order = h["tin"].argsort(stable=True)
    order = order[h["ray"][order].argsort(stable=True)]
    h = {k: x[order] for k, x in h.items()}
    tau = h["sig"] * h["len"]
    run_ = torch.cumsum(tau, 0)
    count = torch.bincount(h["ray"], minlength=R)
    start = torch.cumsum(count, 0) - count
    before = run_ - tau
    before = before - before[start[h["ray"]]]
    on = torch.exp(-before) >= T_MIN
    h = {k: x[on] for k, x in h.items()}
    tau = tau[on]
    t0 = torch.exp(-before[on])
    t1 = t0 * torch.exp(-tau)
    w = t0 - t1
    out = torch.zeros((R, h["q"].shape[1]), device=DEV, dtype=torch.float64)
    out.index_add_(0, h["ray"], w[:, None] * h["q"])
    opac = torch.zeros(R, device=DEV, dtype=torch.float64).index_add_(0, h["ray"], w)
    return out, opac, h, t1, w


def _turn(axis, ang, v):
    """v (R, 3) turned about the unit axis by the angles ang (R)."""
    k = torch.tensor(axis, device=DEV, dtype=torch.float64).expand_as(v)
    s, c = torch.sin(ang)[:, None], torch.cos(ang)[:, None]
    kv = torch.linalg.cross(k, v)
    return v + s * kv + (1.0 - c) * torch.linalg.cross(k, kv)


def _between(p0, p1):
    """Axis and angle of the rotation from pose p0 to pose p1."""
    m = p1[:, :3] @ p0[:, :3].T
    a = 0.5 * np.array([m[2, 1] - m[1, 2], m[0, 2] - m[2, 0], m[1, 0] - m[0, 1]])
    s = np.linalg.norm(a)
    ang = math.atan2(s, 0.5 * (np.trace(m) - 1.0))
    return (a / s if s > 0 else np.array([0.0, 0.0, 1.0])).tolist(), ang


def _rays(sen, lo, hi):
    """Origin, unit direction, time fraction and validity of rays lo..hi of a sensor."""
    i = torch.arange(lo, hi, device=DEV)
    W, H = sen["width"], sen["height"]
    u, v = (i % W).double(), (i // W).double()
    ok = torch.ones(hi - lo, dtype=torch.bool, device=DEV)
    s = torch.zeros_like(u)
    f32 = lambda x: float(np.float32(x))  # noqa: E731  the descriptor holds 32-bit intrinsics
    if sen["kind"] == "lidar":
        e0, e1 = f32(sen["elev_min"]), f32(sen["elev_max"])
        e = e1 - v * ((e1 - e0) / max(1, H - 1))
        a = 2.0 * math.pi * u / W
        d = torch.stack([e.cos() * a.cos(), e.cos() * a.sin(), e.sin()], 1)
        s = u / W
    elif sen["kind"] == "pano":
        e0, e1 = f32(sen["elev_min"]), f32(sen["elev_max"])
        lat = e1 - (v + 0.5) / H * (e1 - e0)
        lon = 2.0 * math.pi * ((u + 0.5) / W - 0.5)
        d = torch.stack([lat.cos() * lon.sin(), -lat.sin(), lat.cos() * lon.cos()], 1)
    else:
        x = (u + 0.5 - f32(sen["cx"])) / f32(sen["fx"])
        y = (v + 0.5 - f32(sen["cy"])) / f32(sen["fy"])
        if sen["kind"] == "pinhole":
            d = torch.stack([x, y, torch.ones_like(x)], 1)
        else:
            th = torch.sqrt(x * x + y * y)
            ok = th <= 0.5 * f32(sen["fov"])
            k = torch.sin(th) / th.clamp_min(1e-300)
            d = torch.stack([k * x, k * y, th.cos()], 1)
    d = d / d.norm(dim=1, keepdim=True)
    p0, p1 = np.asarray(sen["pose0"]), np.asarray(sen["pose1"])
    d = d @ torch.tensor(p0[:, :3].T.copy(), device=DEV)
    axis, ang = _between(p0, p1)
    if ang:
        d = _turn(axis, s * ang, d)
    t0, t1 = torch.tensor(p0[:, 3].copy(), device=DEV), torch.tensor(p1[:, 3].copy(), device=DEV)
    return t0 + s[:, None] * (t1 - t0), d, s, ok


def _frame(grid, sen, cars=(), keep=None, chunk=1 << 20):
    """The sensor's outputs in 64 bits, chunk by chunk; keep(first ray, sums, opacity, hits,
    transmittance after, weights) sees each chunk's hits."""
    R = sen["width"] * sen["height"]
    lidar = sen["kind"] == "lidar"
    sums, opac = [], []
    for lo in range(0, R, chunk):
        hi = min(R, lo + chunk)
        o, d, s, ok = _rays(sen, lo, hi)
        tn = torch.zeros(hi - lo, device=DEV, dtype=torch.float64)
        tf = torch.where(ok, math.inf, -1.0).double()
        found = [grid.field(o, d, *grid.hits(o, d, tn, tf), intensity=lidar)]
        for g, p0, p1 in cars:
            axis, ang = _between(p0, p1)
            a, b = (torch.tensor(p[:, 3].copy(), device=DEV) for p in (p0, p1))
            oa, da = o - (a + s[:, None] * (b - a)), d
            if ang:
                oa, da = _turn(axis, -s * ang, oa), _turn(axis, -s * ang, da)
            r0 = torch.tensor(p0[:, :3].copy(), device=DEV)
            oa, da = oa @ r0, da @ r0
            found.append(g.field(oa, da, *g.hits(oa, da, tn, tf), intensity=lidar))
        h = {k: torch.cat([f[k] for f in found]) for k in found[0]}
        q, op, h, t1, w = _composite(h, hi - lo)
        if keep is not None:
            keep(lo, q, op, h, t1, w)
        sums.append(q)
        opac.append(op)
    q, op = torch.cat(sums), torch.cat(opac)
    out = dict(rgb=q[:, 0:3], depth=q[:, 3], opacity=op)
    if lidar:
        out["intensity"] = q[:, 4]
    return out


def _adjoint(grid, grads, h, t1, w, gq):
    """Adds the adjoint of one chunk's hits to grads: gq (R, columns of q) is dL/d(sums) with the
    opacity's in the last place."""
    g = gq[h["ray"]]
    q = torch.cat([h["q"], torch.ones_like(w)[:, None]], 1)
    wq = w * (g * q).sum(1)
    c = torch.cumsum(wq, 0)
    ends = torch.cumsum(torch.bincount(h["ray"], minlength=gq.shape[0]), 0)
    suffix = c[ends[h["ray"]] - 1] - c
    dsig = (t1 * (g * q).sum(1) - suffix) * h["len"]
    p = grid.params[h["v"]]
    row = torch.zeros((w.shape[0], 32), device=DEV, dtype=torch.float64)
    if grid.mode == "exp":
        gs = dsig * h["sig"]
    else:
        a, b = p[:, 25], p[:, 26]
        e = torch.exp(-h["lin"].abs() / b)
        gs = dsig * a / (2.0 * b) * e
        row[:, 25] = dsig * h["sig"] / a
        row[:, 26] = -dsig * a * h["lin"] * e / (2.0 * b * b)
    row[:, 0:3] = gs[:, None] * h["x"]
    row[:, 3] = gs
    col = h["q"][:, 0:3]
    dz = w[:, None] * g[:, 0:3] * col * (1.0 - col)
    row[:, 4:13] = (dz[:, :, None] * h["x"][:, None]).reshape(-1, 9)
    row[:, 13:25] = (dz[:, :, None] * h["gam"][:, None]).reshape(-1, 12)
    if h["q"].shape[1] > 4:
        i = h["q"][:, 4]
        di = w * g[:, 4] * i * (1.0 - i)
        row[:, 27:30] = di[:, None] * h["x"]
        row[:, 30] = di
    grads.index_add_(0, h["v"], row)


def _exact_regularise(vox, lam_s, lam_a, lam_n):
    """Loss and gradient over the face-adjacent pairs, each counted by its smaller voxel or, at
    equal size, by the one on the lower side."""
    grid = _Grid(vox, "f32")
    p = grid.params.clone().requires_grad_(True)
    n = p.shape[0]
    lo, edge = grid.box(torch.arange(n, device=DEV))
    loss = 0.0
    dims = torch.tensor(grid.dims, device=DEV)
    fine = (lo / (0.5 * grid.s0)).round().long()          # min corner, 0.1 m cells
    size = (edge / (0.5 * grid.s0)).round().long()
    for ax in range(3):
        for sgn in (-1, 1):
            c = fine.clone()
            c[:, ax] = fine[:, ax] + (size if sgn > 0 else -1)
            i = ((c >= 0) & (c < 2 * dims)).all(1).nonzero()[:, 0]
            cell = c[i] >> 1
            e = grid.table[(cell[:, 2] * dims[1] + cell[:, 1]) * dims[0] + cell[:, 0]].long()
            k = c[i] & 1
            kid = grid.kids[(-2 - e).clamp_min(0), k[:, 0] | k[:, 1] << 1 | k[:, 2] << 2]
            j = torch.where(e >= -1, e, kid)
            i, j = i[j >= 0], j[j >= 0]
            on = (size[j] > size[i]) | ((size[j] == size[i]) & (sgn > 0))
            i, j = i[on], j[on]
            X = lo[i] + 0.5 * edge[i][:, None]
            X[:, ax] = lo[i][:, ax] + (edge[i] if sgn > 0 else 0.0)
            ell = edge[i]

            def side(v):
                x = (X - lo[v]) / (0.5 * edge[v][:, None]) - 1.0
                q = p[v]
                s = (q[:, 0:3] * x).sum(1) + q[:, 3]
                if grid.mode == "exp":
                    sig = s.exp()
                else:
                    sig = 0.5 * q[:, 25] * (1.0 + s.sign() * (1.0 - torch.exp(-s.abs() / q[:, 26])))
                return s, 1.0 - torch.exp(-sig * ell), q[:, 0:3] / q[:, 0:3].norm(dim=1, keepdim=True)

            (si, ai, ni), (sj, aj, nj) = side(i), side(j)
            loss = loss + (lam_s * (si - sj).abs() + lam_a * (ai - aj).abs()
                           + lam_n * (1.0 - (ni * nj).sum(1))).sum()
    grads, = torch.autograd.grad(loss, p)
    return dict(loss=loss.detach().reshape(1), grads=grads)


def _exact_densify(st):
    vox = st["vox"]
    p = vox.params.double()
    act = torch.where(st["max_alpha"] < 1e-3, 0, 1)
    l1 = st["grads"][:, 4:13]
    acc = l1[:, 0].abs()
    for k in range(1, 9):                     # the sum that is compared is one of 32-bit terms
        acc = acc + l1[:, k].abs()
    split = (act == 1) & (vox.level < vox.max_level) & (acc > st["threshold"])
    act = torch.where(split, 8, act)
    src = torch.arange(p.shape[0], device=DEV).repeat_interleave(act)
    first = torch.cumsum(act, 0) - act
    child = torch.arange(src.shape[0], device=DEV) - first[src]
    up = split[src]
    s = torch.stack([(child >> a & 1) * 2.0 - 1.0 for a in range(3)], 1).double()
    q = p[src]
    r = q.clone()
    r[:, 3] = q[:, 3] + 0.5 * (q[:, 0:3] * s).sum(1)
    r[:, 0:3] = 0.5 * q[:, 0:3]
    for k in range(3):
        r[:, 13 + 4 * k] += 0.5 * (q[:, 4 + 3 * k:7 + 3 * k] * s).sum(1) / C0
    r[:, 4:13] = 0.5 * q[:, 4:13]
    r[:, 30] = q[:, 30] + 0.5 * (q[:, 27:30] * s).sum(1)
    r[:, 27:30] = 0.5 * q[:, 27:30]
    return dict(level=None, ijk=None, params=torch.where(up[:, None], r, q), counts=None,
                records=None, cells=None, nodes=None)


def _exact_reflect(case, seed):
    st = prepare(case, seed)                 # the first frame's depth and opacity are inputs here
    grid = _Grid(st["vox"], case["dtype"])
    sen = st["sensors"][0]
    D, O = st["depth"].double(), st["opacity"].double()
    o, d, _, _ = _rays(sen, 0, D.numel())
    on = st["opacity"] >= 0.5
    X = o + (D / O.clamp_min(1e-30))[:, None] * d
    g = (X - grid.origin) / grid.s0
    c = torch.floor(g).long()
    dims = torch.tensor(grid.dims, device=DEV)
    on &= ((c >= 0) & (c < dims)).all(1)
    c = torch.minimum(torch.maximum(c, torch.zeros_like(c)), dims - 1)
    e = grid.table[(c[:, 2] * dims[1] + c[:, 1]) * dims[0] + c[:, 0]].long()
    k = (g - c >= 0.5).long()
    v = torch.where(e >= -1, e, grid.kids[(-2 - e).clamp_min(0),
                                          k[:, 0] | k[:, 1] << 1 | k[:, 2] << 2])
    on &= v >= 0
    n = -grid.params[v.clamp_min(0), 0:3]
    n = n / n.norm(dim=1, keepdim=True).clamp_min(1e-300)
    dn = (n * d).sum(1, keepdim=True)
    n, dn = torch.where(dn > 0, -n, n), -dn.abs()
    to = d - 2.0 * dn * n
    rays = torch.zeros((D.numel(), 8), device=DEV, dtype=torch.float64)
    rays[on, 0:3] = (X + 1e-3 * n)[on]
    rays[on, 3:6] = to[on]
    q, op = [], []
    for lo in range(0, rays.shape[0], 1 << 20):
        b = rays[lo:lo + (1 << 20)]
        ok = (b[:, 3:6] != 0).any(1)
        # rays travel as 32-bit numbers
        ro, rd = b[:, 0:3].float().double(), b[:, 3:6].float().double()
        rd = rd / rd.norm(dim=1, keepdim=True).clamp_min(1e-300)
        tn = torch.zeros_like(ro[:, 0])
        h = grid.field(ro, rd, *grid.hits(ro, rd, tn, torch.where(ok, math.inf, -1.0).double()))
        a, w, *_ = _composite(h, b.shape[0])
        q.append(a)
        op.append(w)
    q, op = torch.cat(q), torch.cat(op)
    return dict(rgb=q[:, 0:3], depth=q[:, 3], opacity=op, valid=None, rays=rays)


def exact(case, seed):
    path = case["path"]
    if path == "regularise":
        return _exact_regularise(_voxels(case, seed), 0.01, 0.02, 0.03)
    if path == "densify":
        return _exact_densify(prepare(case, seed))
    if path == "reflect":
        return _exact_reflect(case, seed)
    vox = _voxels(case, seed)
    grid = _Grid(vox, case["dtype"])
    sensors = _sensors(case, seed)
    if path == "serve":
        outs = []
        for s in sensors:
            got = _frame(grid, s)
            outs.append([got[k] for k in _wants(s["kind"])["outputs"]])
        return outs
    if path == "train":
        g = _gen(seed, 3)
        grads = torch.zeros((vox.params.shape[0], 32), device=DEV, dtype=torch.float64)
        R = case["w"] * case["h"]
        targets = [torch.rand((R, 3), generator=g, device=DEV).double() for _ in sensors]
        loss, rgb = 0.0, []
        for s, t in zip(sensors, targets):
            def keep(lo, q, op, h, t1, w, t=t):
                gq = torch.zeros((q.shape[0], 5), device=DEV, dtype=torch.float64)
                gq[:, 0:3] = 2.0 / (3 * R) * (q[:, 0:3] - t[lo:lo + q.shape[0]])
                _adjoint(grid, grads, h, t1, w, gq)
            out = _frame(grid, s, keep=keep)
            loss = loss + ((out["rgb"] - t) ** 2).mean()
            rgb.append(out["rgb"])
        return dict(loss=loss, grads=grads, rgb=rgb)
    sen = sensors[0]
    if path == "lidar_fit":
        g = _gen(seed, 3)
        R = case["w"] * case["h"]
        dg, og, ig = [(torch.randn(R, generator=g, device=DEV) / R).double() for _ in range(3)]
        grads = torch.zeros((vox.params.shape[0], 32), device=DEV, dtype=torch.float64)

        def keep(lo, q, op, h, t1, w):
            at = slice(lo, lo + q.shape[0])
            z = torch.zeros((q.shape[0], 3), device=DEV, dtype=torch.float64)
            gq = torch.cat([z, dg[at, None], ig[at, None], og[at, None]], 1)
            _adjoint(grid, grads, h, t1, w, gq)
        out = _frame(grid, sen, keep=keep)
        out["grads"] = grads
    elif path == "actors":
        cars = [(_Grid(v, case["dtype"]), p0, p1) for v, p0, p1 in _traffic(case, seed)]
        out = _frame(grid, sen, cars)
    else:
        out = _frame(grid, sen)
    names = _wants(sen["kind"])["outputs"] + (("grads",) if path == "lidar_fit" else ())
    return dict({k: out[k] for k in names}, valid=None)
