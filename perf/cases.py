"""The workloads this framework's speed is measured on.

Every case is one pass of a robot's (or a fleet's) map update through the public
entry points: the map follows the robot (``shift``), one frame of the robot's
sensors is fused, and the caller reads the layers it plans on.  A robot's frames
come from a short recorded loop that ``run`` cycles through; its map already
holds an estimate (a stream is under way) with some empty cells and some stale
obstacles, and two boxes move from frame to frame, so every frame has cells to
clear.

  listed()              the cases
  draw(rng)             one more case of the same ranges
  prepare(case, seed)   maps, clouds and read-back buffers, from the seed alone
  run(state)            one pass; returns the layers the caller reads
  work(case)            bytes and operations a pass cannot do without
  exact(case, seed)     the same layers in 64 bits, plain torch
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2204_12876_gb300 import em

RES = 0.04          # metres per cell, every configuration of this repository
FRAMES = 3          # frames in a robot's loop
T_PRIOR = 10        # updates the prior map has seen

DEPTH = dict(noise_a0=0.005, noise_a2=0.002, min_range=0.05, max_range=10.0)
LIDAR = dict(noise_a0=0.01, noise_a2=0.001, min_range=0.3, max_range=40.0)

# layers a planner reads
READ = em.LAYER_ELEVATION | em.LAYER_VARIANCE | em.LAYER_TIME
NORMALS = em.LAYER_NORMAL_X | em.LAYER_NORMAL_Y | em.LAYER_NORMAL_Z


def _case(name=None, kind="map", sensor="depth", points=76800, clouds=1, width=200, height=200, stride=3, ray=True,
          smooth="", paper=False, wall=0, time_variance=0.0, robots=1, mix=0):
    c = dict(kind=kind, sensor=sensor, points=points, clouds=clouds, width=width, height=height, stride=stride,
             ray=ray, smooth=smooth, paper=paper, wall=wall, time_variance=time_variance, robots=robots, mix=mix)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one scattered cloud on a 4 m map, fusion only (the single-update configuration)
        _case("single_20k", sensor="scatter", points=20000, width=100, height=100, ray=False),
        # a filtered depth camera as the paper's rate table has it: few points, 10 m map, ray casting
        _case("camera_6k", points=6276, width=250, height=250),
        # the paper's full pipeline on two dome LiDARs: drift compensation, normals and the guard that reads them,
        # exclusion area, overlap clearance
        _case("domes_43k", sensor="dome", points=21509, clouds=2, width=250, height=250, paper=True),
        # the quadruped's four depth cameras (the depth-stream configuration)
        _case("depth_stream", points=76800, clouds=4, width=200, height=200),
        # one raw 848 x 480 depth image, padded points, wall rule and time variance on: dense cells
        _case("depth_raw_407k", points=407040, width=250, height=250, stride=4, wall=12, time_variance=1e-6),
        # a 128-beam LiDAR on the 20 m map, fusion and ray casting
        _case("lidar_262k", sensor="lidar", points=262144, width=500, height=500),
        # the same with every per-cell feature (the LiDAR configuration)
        _case("lidar_filters", sensor="lidar", points=262144, width=500, height=500, smooth="box", paper=True),
        # a real-time loop whose layers live in the caller's own tensors
        _case("noalloc_depth", kind="noalloc", points=76800, width=200, height=200),
        # one camera whose points and layers live in host memory
        _case("host_camera", kind="host", points=76800, width=200, height=200),
        # 64 uneven maps in one batched update (the batched configuration): points in random order
        _case("batch_64", kind="batch", sensor="scatter", points=400000, width=500, height=500, robots=64, mix=4),
        # one round of the 32-robot fleet through the server, clouds and read-backs on the device
        _case("served_round", kind="server", sensor="mixed", points=262144, width=500, height=500, robots=32, mix=5),
        # a smaller fleet whose clouds and read-backs are in page-locked host memory
        _case("served_host", kind="server_host", sensor="mixed", points=131072, width=350, height=350, robots=12, mix=6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["map", "map", "map", "map", "noalloc", "host", "batch", "batch", "server", "server_host"])
    if kind in ("map", "host"):
        sensor = rng.choice(["depth", "depth", "lidar", "dome", "scatter"])
        clouds = rng.choice([1, 1, 2, 4]) if sensor != "scatter" else 1
        extras = rng.random() < 0.3
        return _case(kind=kind, sensor=sensor, points=_log(rng, 5000, 400000 // clouds), clouds=clouds,
                     width=_log(rng, 100, 500), height=_log(rng, 100, 500), stride=rng.choice([3, 3, 4]),
                     ray=extras or rng.random() < 0.85, paper=extras,
                     smooth=rng.choice(["box", "median", "gauss", ""]) if extras else "",
                     wall=rng.choice([0, 0, 12]), time_variance=rng.choice([0.0, 1e-6]))
    if kind == "noalloc":
        return _case(kind=kind, sensor=rng.choice(["depth", "scatter"]), points=_log(rng, 5000, 300000),
                     width=_log(rng, 64, 256), height=_log(rng, 64, 256), ray=rng.random() < 0.85,
                     time_variance=rng.choice([0.0, 1e-6]))
    most = {"batch": 64, "server": 32, "server_host": 32}[kind]
    return _case(kind=kind, sensor=rng.choice(["mixed", "depth", "scatter"] if kind == "batch" else ["mixed", "depth"]),
                 points=_log(rng, 20000, 262144), width=_log(rng, 120, 500), height=_log(rng, 120, 500),
                 robots=_log(rng, 2, most), mix=rng.randrange(1 << 20))


def _robots(case):
    """One sub-case per robot: sizes and loads of a fleet are uneven."""
    if case["kind"] not in ("batch", "server", "server_host"):
        return [case]
    rng = random.Random(case["mix"])
    out = []
    for i in range(case["robots"]):
        sensor, points = case["sensor"], case["points"]
        if sensor == "mixed":  # half depth cameras, half LiDARs
            sensor = "depth" if i < case["robots"] // 2 else "lidar"
            points = max(2000, points * 76800 // 262144) if sensor == "depth" else points
        elif sensor == "scatter":
            points = rng.randint(min(10000, points), points)
        lo = min(100 if case["kind"] == "batch" else 200, case["width"], case["height"])
        side = rng.randint(lo, max(case["width"], case["height"]))
        square = case["width"] == case["height"]
        out.append(dict(case, sensor=sensor, points=points, width=side,
                        height=side if square else rng.randint(lo, max(case["width"], case["height"]))))
    return out


def _params(case):
    p = dict(width=case["width"], height=case["height"], resolution=RES, var_min=1e-8, mahalanobis_k=2.5,
             outlier_variance=1e-4, ray_step=RES if case["ray"] else 0.0, wall_num_thresh=case["wall"],
             time_variance=case["time_variance"])
    p.update(LIDAR if case["sensor"] in ("lidar", "dome") else DEPTH)
    if case["sensor"] == "scatter":
        p.update(min_range=0.0, max_range=1e9)
    if case["paper"]:
        p.update(flags=em.F_NORMALS, drift_flatness=0.95, cleanup_normal_thresh=0.1, excl_b=0.3, excl_c=0.5,
                 excl_theta=0.6, excl_d=1.5, overlap_radius=0.6, overlap_dz=1.5)
    if case["smooth"]:
        p["flags"] = p.get("flags", 0) | em.F_INPAINT | em.F_UPPER | {
            "box": em.F_SMOOTH, "median": em.F_MEDIAN, "gauss": em.F_GAUSS}[case["smooth"]]
    return p


def _mask(case):
    mask = READ
    if case["paper"]:
        mask |= NORMALS
    if case["smooth"]:
        mask |= em.LAYER_SMOOTH | em.LAYER_INPAINT | em.LAYER_UPPER
    return mask


def _layers(mask):
    return bin(mask).count("1")


# ---------------------------------------------------------------- inputs

class _Scene:
    """A height field: three sinusoids, a step, boxes, stairs for the LiDAR, two boxes that move."""

    HALF, STEP = 16.0, 0.04

    def __init__(self, seed, stairs):
        rng = np.random.default_rng(seed)
        n = int(2 * self.HALF / self.STEP) + 1
        ax = torch.linspace(-self.HALF, self.HALF, n, device="cuda")
        y, x = torch.meshgrid(ax, ax, indexing="ij")
        z = torch.zeros_like(x)
        amp = (0.03 if stairs else 0.2) * rng.dirichlet(np.ones(3))
        for a in amp:
            lam, ang, ph = rng.uniform(0.5, 4.0), rng.uniform(0, 2 * math.pi), rng.uniform(0, 2 * math.pi)
            z += float(a) * torch.sin((2 * math.pi / lam) * (math.cos(ang) * x + math.sin(ang) * y) + ph)
        a = rng.uniform(0, 2 * math.pi)
        z += 0.15 * ((math.cos(a) * x + math.sin(a) * y) > rng.uniform(-1.5, 1.5))
        if stairs:  # ten stairs (0.17 m rise, 0.30 m run) and a 15 degree ramp
            xs, ys = rng.uniform(1.5, 3.0), rng.uniform(-1.0, 1.0)
            k = torch.clamp(torch.floor((x - xs) / 0.3) + 1, 0, 10)
            z += torch.where(((y - ys).abs() <= 1.5) & (x < xs + 5.0), 0.17 * k, torch.zeros_like(k))
            xr, yr = -2.0 - rng.uniform(0, 1), rng.uniform(3.0, 4.0)
            ramp = torch.clamp(xr - x, 0.0, 6.0) * math.tan(math.radians(15.0))
            z += torch.where((y >= yr) & (y <= yr + 4.0), ramp, torch.zeros_like(ramp))
        for _ in range(30):
            self._box(z, *rng.uniform(-5, 5, 2), *rng.uniform(0.05, 0.3, 2), rng.uniform(0.05, 0.4))
        self.ground, self.walk = z, rng.uniform(-2.5, 2.5, (2, 2))
        self.step_xy, self.tall = rng.normal(0, 0.25, (2, 2)), rng.uniform(0.4, 0.9, 2)
        self.field = z

    def _box(self, z, cx, cy, hx, hy, tall):
        i = [int(round((v + self.HALF) / self.STEP)) for v in (cx - hx, cx + hx, cy - hy, cy + hy)]
        part = z[i[2]:i[3] + 1, i[0]:i[1] + 1]
        if part.numel():
            part.copy_(torch.maximum(part, part.min() + float(tall)))

    def frame(self, k):
        """The scene at frame k of the loop."""
        self.field = self.ground.clone()
        for b in range(2):
            cx, cy = self.walk[b] + k * self.step_xy[b]
            self._box(self.field, cx, cy, 0.2, 0.2, self.tall[b])

    def height(self, x, y):
        grid = torch.stack([x, y], dim=-1).reshape(1, 1, -1, 2) / self.HALF
        return torch.nn.functional.grid_sample(self.field[None, None], grid, mode="bilinear", padding_mode="border",
                                               align_corners=True).reshape(x.shape)

    def cast(self, o, d, far):
        """Distance to the surface along unit rays from o, NaN beyond `far`."""
        o = torch.tensor(o, dtype=torch.float32, device="cuda")
        above = lambda t: o[2] + t * d[:, 2] - self.height(o[0] + t * d[:, 0], o[1] + t * d[:, 1])  # noqa: E731
        t = 0.05 * (far / 0.05) ** torch.linspace(0.0, 1.0, 288, device="cuda")
        under = above(t[:, None].expand(-1, d.shape[0])) <= 0  # (steps, rays)
        miss = ~under.any(dim=0)
        first = under.to(torch.uint8).argmax(dim=0)
        hi = t[first]
        lo = torch.where(first > 0, t[(first - 1).clamp(min=0)], torch.zeros_like(hi))
        for _ in range(14):
            mid = 0.5 * (lo + hi)
            low = above(mid) <= 0
            hi = torch.where(low, mid, hi)
            lo = torch.where(low, lo, mid)
        return torch.where(miss, torch.full_like(hi, math.nan), hi)


def _rot_z(a):
    c, s = math.cos(a), math.sin(a)
    return np.array([[c, -s, 0.0], [s, c, 0.0], [0.0, 0.0, 1.0]])


def _pose(R, t):
    return np.concatenate([R, np.asarray(t, np.float64)[:, None]], axis=1).astype(np.float32).reshape(12)


def _depth_dirs(n):
    """Pixel directions (optical frame, z = 1) of an image of about 4:3 with n pixels, the last row cut."""
    w = max(8, int(round(math.sqrt(n * 4 / 3))))
    h = (n + w - 1) // w
    f = 200.0 * w / 320.0
    v, u = torch.meshgrid(torch.arange(h, device="cuda") + 0.5, torch.arange(w, device="cuda") + 0.5, indexing="ij")
    d = torch.stack([(u - w / 2) / f, (v - h / 2) / f, torch.ones_like(u)], dim=-1).reshape(-1, 3)
    return d[:n].contiguous()


def _scan_dirs(n, beams, lo_deg, hi_deg):
    """Unit directions of a spinning scan, beam by beam, n points."""
    az = (n + beams - 1) // beams
    e = torch.deg2rad(torch.linspace(lo_deg, hi_deg, beams, device="cuda"))
    a = torch.arange(az, device="cuda") * (2 * math.pi / az)
    E, A = torch.meshgrid(e, a, indexing="ij")
    d = torch.stack([torch.cos(E) * torch.cos(A), torch.cos(E) * torch.sin(A), torch.sin(E)], dim=-1).reshape(-1, 3)
    return d[:n].contiguous()


def _cloud(case, scene, body, yaw, k, gen):
    """Cloud k of the robot: (points (n, stride) float32 on the GPU, pose)."""
    n = case["points"]
    noise = torch.randn(n, device="cuda", generator=gen)
    if case["sensor"] == "scatter":  # uniform over the map and a little beyond, no occlusion, random order
        half = [0.5 * RES * 1.05 * case[s] for s in ("width", "height")]
        u = torch.rand(2, n, device="cuda", generator=gen) * 2 - 1
        x, y = u[0] * half[0], u[1] * half[1]
        z = scene.height(x, y)
        R, t = _rot_z(yaw), np.array([0.0, 0.0, 0.5])
        dz = 0.5 - z
        p = torch.stack([x, y, z + noise * (0.005 + 0.002 * dz * dz)], dim=1) - torch.tensor(
            t, dtype=torch.float32, device="cuda")
        p = p @ torch.tensor(R, dtype=torch.float32, device="cuda")
    elif case["sensor"] == "depth":  # pinhole camera pitched 40 degrees down, 0.3 m from the body's centre
        th = math.radians(40.0)
        zf, xr = np.array([math.cos(th), 0.0, -math.sin(th)]), np.array([0.0, -1.0, 0.0])
        R = _rot_z(yaw + k * math.pi / 2) @ np.stack([xr, np.cross(zf, xr), zf], axis=1)
        t = body + _rot_z(yaw + k * math.pi / 2) @ np.array([0.3, 0.0, 0.0])
        dirs = _depth_dirs(n)
        norm = dirs.norm(dim=1)
        depth = scene.cast(t, (dirs / norm[:, None]) @ torch.tensor(R.T, dtype=torch.float32, device="cuda"), 11.0) / norm
        depth = torch.where(depth > 8.0, torch.full_like(depth, math.nan), depth)
        depth = depth + noise * (0.005 + 0.002 * depth * depth)
        p = dirs * depth[:, None]
        p[torch.rand(n, device="cuda", generator=gen) < 0.05] = math.nan  # dropped pixels
    else:
        if case["sensor"] == "lidar":
            R, t, dirs = _rot_z(yaw), body + np.array([0.0, 0.0, 0.1]), _scan_dirs(n, min(128, max(16, n // 512)), -45.0, 15.0)
        else:  # dome LiDARs at the front and the back, a hemisphere each
            R, t = _rot_z(yaw + k * math.pi), body + _rot_z(yaw + k * math.pi) @ np.array([0.35, 0.0, 0.0])
            dirs = _scan_dirs(n, 32, -88.0, 2.0)
        r = scene.cast(t, dirs @ torch.tensor(R.T, dtype=torch.float32, device="cuda"), 30.0)
        r = r + noise * (0.01 + 0.001 * r * r)
        p = dirs * r[:, None]
    if case["stride"] == 4:
        p = torch.cat([p, torch.zeros(n, 1, device="cuda")], dim=1)
    return p.contiguous(), _pose(R, t)


class _Robot:
    """One robot's recorded loop and its map's prior state."""

    def __init__(self, case, seed):
        self.case = case
        rng = np.random.default_rng([seed, 17])
        gen = torch.Generator(device="cuda")
        gen.manual_seed(int(rng.integers(1 << 62)))
        scene = _Scene([seed, 23], case["sensor"] in ("lidar", "dome"))
        W, H = case["width"], case["height"]
        # prior: terrain at the cell centres, 15 % empty, 3 % stale obstacles
        xs = (torch.arange(W, device="cuda") + 0.5 - W / 2) * RES
        ys = (torch.arange(H, device="cuda") + 0.5 - H / 2) * RES
        Y, X = torch.meshgrid(ys, xs, indexing="ij")
        rand = lambda: torch.rand(H, W, device="cuda", generator=gen)  # noqa: E731
        h = scene.height(X, Y) + 0.01 * torch.randn(H, W, device="cuda", generator=gen)
        h = torch.where(rand() < 0.03, h + 0.1 + 0.4 * rand(), h)
        var = 10.0 ** (rand() * 2 - 5)
        empty = rand() < 0.15
        h[empty], var[empty] = math.nan, math.inf
        self.prior = {"h": h, "var": var, "t": torch.floor(rand() * T_PRIOR)}
        if case["paper"]:
            n = torch.stack([0.2 * torch.randn(H, W, device="cuda", generator=gen),
                             0.2 * torch.randn(H, W, device="cuda", generator=gen), torch.ones(H, W, device="cuda")])
            n = n / n.norm(dim=0)
            n[:, (rand() < 0.1) | empty] = math.nan
            self.prior.update(nx=n[0], ny=n[1], nz=n[2])
        self.frames, self.shifts = [], []
        xy, yaw = np.zeros(2), float(rng.uniform(0, 2 * math.pi))
        for k in range(FRAMES):
            if case["sensor"] != "scatter":  # a walking robot
                xy = xy + rng.normal(0.0, 0.03, 2)
                yaw += math.radians(rng.normal(0.0, 1.0))
            scene.frame(k)
            p0 = torch.tensor([xy[0]], dtype=torch.float32, device="cuda")
            p1 = torch.tensor([xy[1]], dtype=torch.float32, device="cuda")
            body = np.array([xy[0], xy[1], float(scene.height(p0, p1)) + 0.5])
            self.frames.append([_cloud(case, scene, body, yaw, c, gen) for c in range(case["clouds"])])
            self.shifts.append((int(round(xy[0] / RES)), int(round(xy[1] / RES))))

    def load(self, m):
        """Put the prior state into a map."""
        names = ["h", "var", "t"] + (["nx", "ny", "nz"] if "nx" in self.prior else [])
        m.set_layers(READ | (NORMALS if "nx" in self.prior else 0), torch.stack([self.prior[n] for n in names]))
        m.set_state(t_now=T_PRIOR)


def _seeds(case, seed):
    return [seed * 1009 + i for i in range(len(_robots(case)))]


# ---------------------------------------------------------------- one map

class _MapState:
    """One robot, one resident map: Map.shift, Map.update / update_multi, Map.get_layers."""

    def __init__(self, case, seed):
        r = _Robot(case, _seeds(case, seed)[0])
        self.frames, self.shifts = r.frames, r.shifts
        self.map = em.Map(em.Params(**_params(case)))
        self.map.reserve(case["points"] * case["clouds"])
        r.load(self.map)
        self.mask = _mask(case)
        self.out = torch.empty(_layers(self.mask), case["height"], case["width"], device="cuda")
        self.layers = list(self.out.unbind(0))
        self.at, self.k = (0, 0), 0
        torch.cuda.synchronize()

    def follow(self):
        x, y = self.shifts[self.k % FRAMES]
        if (x, y) != self.at:
            self.map.shift(x - self.at[0], y - self.at[1])
            self.at = (x, y)

    def run(self):
        self.follow()
        clouds = self.frames[self.k % FRAMES]
        if len(clouds) == 1:
            self.map.update(*clouds[0])
        else:
            self.map.update_multi(clouds)
        self.k += 1
        self.map.get_layers(self.mask, out=self.out)
        return self.layers


class _HostState(_MapState):
    """The same with the clouds and the layers in host memory: Map.update_host, host get_layers."""

    def __init__(self, case, seed):
        super().__init__(case, seed)
        self.frames = [[(p.cpu().numpy(), q) for p, q in f] for f in self.frames]

    def run(self):
        self.follow()
        self.map.update_host(self.frames[self.k % FRAMES])
        self.k += 1
        return list(self.map.get_layers(self.mask))


class _NoallocState:
    """A caller that owns its layers: update_noalloc on tensors of its own (the map stands still)."""

    def __init__(self, case, seed):
        r = _Robot(case, _seeds(case, seed)[0])
        self.frames = r.frames
        self.params = em.Params(**_params(case))
        self.h, self.var = r.prior["h"].contiguous(), r.prior["var"].contiguous()
        self.t = r.prior["t"].to(torch.int32).contiguous()
        self.k = 0
        torch.cuda.synchronize()

    def run(self):
        em.update_noalloc(self.params, self.h, self.var, self.t, self.frames[self.k % FRAMES], t_now=T_PRIOR + 1 + self.k)
        self.k += 1
        return [self.h, self.var, self.t]


# ---------------------------------------------------------------- many maps

class _BatchState:
    """Uneven maps in one update: Batch.update (graph replay), then every map's layers."""

    def __init__(self, case, seed):
        subs = _robots(case)
        robots = [_Robot(c, s) for c, s in zip(subs, _seeds(case, seed))]
        self.maps = [em.Map(em.Params(**_params(c))) for c in subs]
        for r, m in zip(robots, self.maps):
            r.load(m)
        self.batch = em.Batch(max_maps=len(subs), max_clouds=len(subs), max_points=sum(c["points"] for c in subs),
                              max_cells=max(c["width"] * c["height"] for c in subs))
        self.pairs = [[(m, *r.frames[k][0]) for r, m in zip(robots, self.maps)] for k in range(FRAMES)]
        cells = [c["width"] * c["height"] for c in subs]
        self.out = torch.empty(2 * sum(cells), device="cuda")
        self.parts = list(torch.split(self.out, [2 * n for n in cells]))
        self.k = 0
        torch.cuda.synchronize()

    def run(self):
        self.batch.update(self.pairs[self.k % FRAMES])
        self.k += 1
        for m, o in zip(self.maps, self.parts):
            m.get_layers(em.LAYER_ELEVATION | em.LAYER_VARIANCE, out=o)
        return self.out


class _ServerState:
    """A fleet's round: Server.submit_many with read-backs, then wait_many."""

    def __init__(self, case, seed):
        subs = _robots(case)
        host = case["kind"] == "server_host"
        robots = [_Robot(c, s) for c, s in zip(subs, _seeds(case, seed))]
        cells = [c["width"] * c["height"] for c in subs]
        self.server = em.Server(budget_bytes=40 << 30, max_slots=4096, n_streams=3,
                                max_batch_maps=min(16, len(subs)), max_batch_points=sum(c["points"] for c in subs),
                                max_map_cells=max(cells))
        self.ids = [self.server.add_map(em.Params(**_params(c))) for c in subs]
        for r, i in zip(robots, self.ids):
            r.load(self.server.map(i))
        place = (lambda p: p.cpu().pin_memory()) if host else (lambda p: p)
        self.clouds = [[(place(r.frames[k][0][0]), r.frames[k][0][1]) for r in robots] for k in range(FRAMES)]
        self.out = place(torch.empty(2 * sum(cells), device="cuda"))
        self.parts = list(torch.split(self.out, [2 * n for n in cells]))
        self.k = 0
        torch.cuda.synchronize()

    def run(self):
        clouds = self.clouds[self.k % FRAMES]
        self.k += 1
        tickets = self.server.submit_many([(i, [c], (em.LAYER_ELEVATION | em.LAYER_VARIANCE, o))
                                           for i, c, o in zip(self.ids, clouds, self.parts)])
        status = self.server.wait_many(tickets)
        if any(status):
            raise RuntimeError(f"requests failed: {status}")
        return self.out


def prepare(case, seed):
    return {"map": _MapState, "host": _HostState, "noalloc": _NoallocState, "batch": _BatchState,
            "server": _ServerState, "server_host": _ServerState}[case["kind"]](case, int(seed))


def run(state):
    return state.run()


def work(case):
    """Every point and every cell's state read once, every layer the caller reads written once."""
    n_bytes = flops = 0.0
    for c in _robots(case):
        points, cells = c["points"] * c["clouds"], c["width"] * c["height"]
        layers = 2 if c["kind"] in ("batch", "server", "server_host") else _layers(_mask(c))
        n_bytes += 4.0 * c["stride"] * points + 12.0 * cells + 4.0 * layers * cells
        flops += 60.0 * points
    return {"bytes": n_bytes, "flops": flops}


# ---------------------------------------------------------------- 64 bits

def _f(v):
    return float(np.float32(v))


def _r32(x):
    """Round to float32, kept as float64."""
    return x.to(torch.float32).to(torch.float64)


def _exact_map(case, robot):
    """h, var and t after the robot's first frame, in 64 bits.  Which cell a point or a ray sample falls into,
    and whether a point or a sample is beyond a threshold, is defined on float32 (points, poses and layers
    are float32), so those decisions round where float32 does; the estimates are summed and divided in 64 bits."""
    P = em.Params(**_params(case))
    W, H, k = P.width, P.height, 0
    dx, dy = robot.shifts[0] if case["kind"] in ("map", "host") else (0, 0)
    t_now = T_PRIOR + 1
    h = torch.full((H, W), math.nan, dtype=torch.float64, device="cuda")
    var = torch.full_like(h, math.inf)
    t = torch.zeros_like(h)
    ys, xs = slice(max(0, dy), min(H, H + dy)), slice(max(0, dx), min(W, W + dx))
    yd, xd = slice(max(0, -dy), min(H, H - dy)), slice(max(0, -dx), min(W, W - dx))
    h[yd, xd], var[yd, xd] = robot.prior["h"][ys, xs].double(), robot.prior["var"][ys, xs].double()
    t[yd, xd] = robot.prior["t"][ys, xs].double()
    res, inv = _f(P.resolution), _f(1.0 / _f(P.resolution))
    x0, y0 = _f(res * (dx - 0.5 * W)), _f(res * (dy - 0.5 * H))
    h, var, t = h.reshape(-1), var.reshape(-1), t.reshape(-1)
    valid = torch.isfinite(var)
    ve = _r32(_f(P.time_variance) * (t_now - t) + var)
    thr = torch.where(valid, _r32(h - _r32(ve.sqrt())), torch.full_like(h, -math.inf))
    cells = W * H
    count = torch.zeros(cells, dtype=torch.int64, device="cuda")
    mark = torch.zeros(cells, dtype=torch.bool, device="cuda")
    rec = []
    z_ref = float(robot.frames[0][0][1][11])
    for pts, pose in robot.frames[0]:
        q = [float(v) for v in pose]
        p = pts[:, :3].double()
        fin = torch.isfinite(p).all(dim=1)
        p = p[fin]
        px, py, pz = p.unbind(dim=1)
        d = _r32(_r32(px * px + _r32(py * py + _r32(pz * pz))).sqrt())
        near = (d >= _f(P.min_range)) & (d <= _f(P.max_range))
        px, py, pz, d = px[near], py[near], pz[near], d[near]
        v = [_r32(q[4 * r] * px + _r32(q[4 * r + 1] * py + _r32(q[4 * r + 2] * pz))) for r in range(3)]
        x, y, z = (_r32(v[r] + q[4 * r + 3]) for r in range(3))
        ix = torch.floor(_r32(_r32(x - x0) * inv))
        iy = torch.floor(_r32(_r32(y - y0) * inv))
        inm = (ix >= 0) & (iy >= 0) & (ix < W) & (iy < H)
        cell = (iy * W + ix)[inm].long()
        s32 = _r32(_r32(_f(P.noise_a2) * d + _f(P.noise_a1)) * d + _f(P.noise_a0))
        vp32 = torch.clamp(_r32(s32 * s32), min=_f(P.var_min))
        d64 = torch.stack([px, py, pz]).square().sum(dim=0).sqrt()
        vp = torch.clamp((_f(P.noise_a0) + _f(P.noise_a1) * d64 + _f(P.noise_a2) * d64 * d64) ** 2, min=_f(P.var_min))
        z64 = q[8] * px + q[9] * py + q[10] * pz + q[11]
        rec.append((cell, z[inm], z64[inm], vp32[inm], vp[inm]))
        count += torch.bincount(cell, minlength=cells)
        if P.ray_step > 0:
            step = _f(P.ray_step)
            c = _r32(step / torch.clamp(d, min=1e-30))
            a = [_r32(_r32(torch.tensor(q[3], dtype=torch.float64) - x0) * inv).item(),
                 _r32(_r32(torch.tensor(q[7], dtype=torch.float64) - y0) * inv).item()]
            b = [_r32(_r32(c * v[r]) * inv) for r in range(2)]
            bz = _r32(c * v[2])
            far = int(min(float(d.max()) / step, 2.0 * math.hypot(W, H))) + 2 if d.numel() else 0
            for k in range(1, far):
                ku = _f(_f(k) * np.float32(step))
                sx, sy = torch.floor(_r32(k * b[0] + a[0])), torch.floor(_r32(k * b[1] + a[1]))
                ok = (ku < d) & (sx >= 0) & (sy >= 0) & (sx < W) & (sy < H) & ~((sx == ix) & (sy == iy))
                at = torch.where(ok, sy * W + sx, torch.zeros_like(sx)).long()
                below = ok & (_r32(k * bz + q[11]) < thr[at])
                mark[at[below]] = True
    cell, z, z64, vp32, vp = (torch.cat(v) for v in zip(*rec))
    cv, ch, cve = valid[cell], h[cell], ve[cell]
    wall = (cv & (count[cell] > P.wall_num_thresh) & (z < ch)) if P.wall_num_thresh > 0 else torch.zeros_like(cv)
    dz = _r32(z - ch)
    kk = _f(_f(P.mahalanobis_k) ** 2)
    rej = cv & ~wall & (_r32(dz * dz) > _r32(kk * _r32(cve + vp32)))
    acc = ~wall & ~rej
    href = torch.where(valid, h, torch.full_like(h, z_ref))
    add = lambda w: torch.zeros(cells, dtype=torch.float64, device="cuda").index_add_(0, cell, w)  # noqa: E731
    zero = torch.zeros_like(vp)
    sw = add(torch.where(acc, 1.0 / vp, zero))
    st = add(torch.where(acc, (z64 - href[cell]) / vp, zero))
    n_acc, n_rej = add(acc.double()), add(rej.double())
    prior = _f(P.time_variance) * (t_now - t) + var + n_rej * _f(P.outlier_variance)
    lam = torch.where(valid, 1.0 / prior, torch.zeros_like(prior)) + sw
    wrote = (n_acc + n_rej) > 0
    h_new = torch.where(n_acc > 0, href + st / lam, h)
    v_new = torch.where(n_acc > 0, 1.0 / lam, prior)
    h, var, t = torch.where(wrote, h_new, h), torch.where(wrote, v_new, var), torch.where(wrote, torch.full_like(t, t_now), t)
    gone = mark & torch.isfinite(var) & (t_now - t >= max(1, P.cleanup_min_age))
    h[gone], var[gone] = math.nan, math.inf
    return h, var, t


def exact(case, seed):
    if case["paper"] or case["smooth"]:  # drift, guard and stencils: float32 definitions all through
        return None
    got = []
    for c, s in zip(_robots(case), _seeds(case, int(seed))):
        got.append(_exact_map(c, _Robot(c, s)))
    h, var, t = got[0]
    shape = (case["height"], case["width"])
    if case["kind"] in ("map", "host"):
        return [v.reshape(shape) for v in (h, var, t)]
    if case["kind"] == "noalloc":
        return [h.reshape(shape), var.reshape(shape), None]
    return torch.cat([v for g in got for v in g[:2]])
