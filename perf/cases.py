"""Workloads of the TSDF library as its users run them, for timing.

Every case is a program's use of the public calls on seeded synthetic input:
a camera, a LiDAR or a rig that feeds a map while it moves, a recorded
sequence fused in one call, several maps served together, the layers derived
from a map.  The scenes are a furnished room (an inward box with boxes and
spheres) and an open lot (a ground plane with boxes and poles), ray-cast on
the GPU with the noise of a depth camera or a LiDAR; sizes are those of the
repository's workloads (64x48 to 1280x720 depth, 1024x64 beams, voxels of 2,
5 and 10 cm, up to 300 frames).  After the integration the map is read back
whole: the voxel centres of every block near a measured surface are looked
up, which returns every voxel that the pass wrote.

`exact` repeats the update rules in FP64 with plain torch: band of each pixel,
projection, truncation, running average.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2311_00626_gb300 as gt

DEV = "cuda"
STORAGE = {"fp32": gt.STORAGE_FP32, "fp16": gt.STORAGE_FP16, "fixed16": gt.STORAGE_FIXED16}
MAX_WEIGHT = 100.0
PIXELS_MOST = 300 * 640 * 480  # the largest listed sequence


def listed():
    return [
        # one 64x48 frame into a live map: the smallest call, all launch and latency
        {"name": "tiny_frame", "kind": "live", "width": 64, "height": 48, "frames": 1, "voxel": 0.05,
         "storage": "fp32", "trunc": 4},
        # a 30 Hz RGB-D camera: eight frames, one call each as they arrive
        {"name": "live_640x480", "kind": "live", "width": 640, "height": 480, "frames": 8, "voxel": 0.02,
         "storage": "fp32", "trunc": 4},
        # the dynamic layer: occupancy from a wide camera, faded after every frame
        {"name": "occupancy_848x480", "kind": "occupancy", "width": 848, "height": 480, "frames": 4,
         "voxel": 0.05, "storage": "fp32", "trunc": 4},
        # a spinning LiDAR: four scans, one call each
        {"name": "lidar_1024x64", "kind": "lidar", "width": 1024, "height": 64, "frames": 4, "voxel": 0.05,
         "storage": "fp32", "trunc": 4},
        # a recorded room sequence fused from scratch in one call
        {"name": "room_300", "kind": "batch", "width": 640, "height": 480, "frames": 300, "voxel": 0.02,
         "storage": "fp32", "trunc": 4, "weighting": 0},
        # high resolution with the sensor-error weights, coarser voxels
        {"name": "weighted_1280x720", "kind": "batch", "width": 1280, "height": 720, "frames": 24,
         "voxel": 0.05, "storage": "fp32", "trunc": 4, "weighting": 1},
        # four cameras and a LiDAR on one vehicle: a call per step, 16-bit voxels
        {"name": "rig_8_steps", "kind": "rig", "frames": 8, "voxel": 0.05, "storage": "fixed16", "trunc": 4},
        # sixteen maps served together, mixed sensors and voxel sizes
        {"name": "serve_16_maps", "kind": "serve", "maps": 16, "frames": 64, "storage": "fp16", "trunc": 4},
        # a recorded sequence in pinned host memory, copied as it is fused
        {"name": "host_96", "kind": "host", "width": 640, "height": 480, "frames": 96, "voxel": 0.02,
         "storage": "fp32", "trunc": 4, "weighting": 0},
        # a colour layer from registered depth and colour images
        {"name": "color_32", "kind": "color", "width": 640, "height": 480, "frames": 32, "voxel": 0.02,
         "storage": "fp32", "trunc": 4},
        # the planner's layer: distances of a fresh map, then brought up to date
        {"name": "esdf_40_plus_8", "kind": "esdf", "width": 640, "height": 480, "frames": 48, "voxel": 0.02,
         "storage": "fp32", "trunc": 4, "first": 40},
        # the surface of a map, in a fixed order
        {"name": "mesh_64", "kind": "mesh", "width": 640, "height": 480, "frames": 64, "voxel": 0.02,
         "storage": "fp32", "trunc": 4, "changed": False},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["live", "live", "occupancy", "lidar", "batch", "batch", "rig", "serve", "host", "color",
                       "esdf", "mesh"])
    c = {"kind": kind, "storage": rng.choice(["fp32", "fp16", "fixed16"]), "trunc": rng.choice([4, 4, 6])}
    if kind == "rig":
        return {**c, "frames": rng.randint(2, 10), "voxel": rng.choice([0.05, 0.1])}
    if kind == "serve":
        return {**c, "maps": rng.randint(2, 16), "frames": rng.randint(16, 80)}
    if kind == "lidar":
        return {**c, "width": log_int(256, 2048), "height": rng.choice([16, 32, 64, 128]),
                "frames": rng.randint(1, 8), "voxel": rng.choice([0.05, 0.1])}
    w = log_int(64, 1280)
    h = max(36, int(w * rng.uniform(0.5, 0.8)))
    c.update(width=w, height=h, voxel=rng.choice([0.02, 0.02, 0.05, 0.1] if w >= 200 else [0.05, 0.1]))
    most = max(1, min(300, PIXELS_MOST // (w * h)))
    if kind in ("live", "occupancy"):
        return {**c, "frames": rng.randint(1, 12)}
    if kind in ("batch", "host"):
        return {**c, "frames": min(most, log_int(5, 300)), "weighting": rng.choice([0, 0, 1, 2, 3])}
    if kind == "color":
        return {**c, "frames": min(most, log_int(2, 48))}
    if kind == "esdf":
        first = log_int(4, 40)
        return {**c, "frames": first + rng.randint(1, 10), "first": first}
    return {**c, "frames": log_int(4, 64), "changed": rng.random() < 0.5}


# ------------------------------------------------------------------ inputs

def _room(rs, path):
    """40 boxes and 20 spheres in a 10x10x3 m room, none within 0.4 m of the path."""
    size = np.array([10.0, 10.0, 3.0])

    def clear(lo, hi):
        gap = np.maximum(np.maximum(lo - path, path - hi), 0.0)
        return np.sqrt((gap ** 2).sum(1)).min() > 0.4

    boxes = []
    while len(boxes) < 40:
        e = rs.uniform(0.2, 1.5, 3)
        c = rs.uniform(0.5 * e, size - 0.5 * e)
        if clear(c - 0.5 * e, c + 0.5 * e):
            boxes.append(np.concatenate([c - 0.5 * e, c + 0.5 * e]))
    balls = []
    while len(balls) < 20:
        r = rs.uniform(0.1, 0.5)
        c = rs.uniform(r, size - r)
        if clear(c - r, c + r):
            balls.append(np.concatenate([c, [r]]))
    return {"room": np.concatenate([np.zeros(3), size]), "boxes": np.stack(boxes), "balls": np.stack(balls)}


def _lot(rs, path):
    """200 boxes and 50 poles on the ground of a 40x40 m lot, none within 0.6 m of the path."""
    boxes = []
    while len(boxes) < 250:
        e = rs.uniform(0.2, 1.5, 3) if len(boxes) < 200 else np.array([0.2, 0.2, rs.uniform(1.0, 5.0)])
        lo = np.array([*rs.uniform(0.0, 40.0 - e[:2]), 0.0])
        gap = np.maximum(np.maximum(lo - path, path - (lo + e)), 0.0)
        if np.sqrt((gap ** 2).sum(1)).min() > 0.6:
            boxes.append(np.concatenate([lo, lo + e]))
    return {"ground": True, "boxes": np.stack(boxes)}


def _path(rs, n, centre, radius, step):
    """n poses (camera axes x right, y down, z forward) on a wavy closed path at
    about 1.5 m height, `step` metres apart, panning and nodding a little."""
    ph = rs.uniform(0, 2 * math.pi, 6)
    s = ph[0] + np.arange(n + 1) * (step / radius)
    r = radius * (1 + 0.12 * np.sin(3 * s + ph[1]))
    p = np.stack([centre + r * np.cos(s), centre + r * np.sin(s), 1.5 + 0.08 * np.sin(2 * s + ph[2])], 1)
    fwd = np.diff(p, axis=0)
    yaw = np.arctan2(fwd[:, 1], fwd[:, 0]) + 0.6 * np.sin(2 * s[:-1] + ph[3])
    pitch = 0.12 * np.sin(3 * s[:-1] + ph[4])
    z = np.stack([np.cos(yaw) * np.cos(pitch), np.sin(yaw) * np.cos(pitch), np.sin(pitch)], 1)
    x = np.stack([np.sin(yaw), -np.cos(yaw), 0 * yaw], 1)
    T = np.zeros((n, 4, 4))
    T[:, :3, 0], T[:, :3, 1], T[:, :3, 2], T[:, :3, 3], T[:, 3, 3] = x, np.cross(z, x), z, p[:-1], 1.0
    return T


def _pinhole(w, h):
    f = 525.0 * w / 640
    return {"kind": "pinhole", "fu": f, "fv": f, "cu": (w - 1) / 2, "cv": (h - 1) / 2, "width": w, "height": h}


def _lidar(n_az, n_el):
    return {"kind": "lidar", "n_az": n_az, "n_el": n_el, "theta_start": -math.pi,
            "phi_start": math.radians(67.5), "el_fov": math.radians(45.0), "min_range": 0.5, "max_range": 30.0}


def _shape(s):
    return (s["height"], s["width"]) if s["kind"] == "pinhole" else (s["n_el"], s["n_az"])


def _f32(x):
    return float(np.float32(x))


def _rays(s, dtype):
    """Ray directions of a sensor's pixels in its own frame, [3][H, W]: z = 1 (camera) or unit length (LiDAR)."""
    h, w = _shape(s)
    j = torch.arange(h, device=DEV, dtype=dtype)[:, None].expand(h, w)
    i = torch.arange(w, device=DEV, dtype=dtype)[None].expand(h, w)
    if s["kind"] == "pinhole":
        return [(i - _f32(s["cu"])) / _f32(s["fu"]), (j - _f32(s["cv"])) / _f32(s["fv"]), torch.ones_like(i)]
    th = _f32(s["theta_start"]) + (i + 0.5) * (2 * math.pi / w)
    ph = _f32(s["phi_start"]) + (j + 0.5) * (_f32(s["el_fov"]) / h)
    return [torch.sin(ph) * torch.cos(th), torch.sin(ph) * torch.sin(th), torch.cos(ph)]


def _cast(scenes, s, Ts, gen):
    """Depth or range images [F, H, W] of sensor s at poses Ts, frame f in scenes[f], with the sensor's noise."""
    F, (h, w) = len(Ts), _shape(s)
    out = torch.empty((F, h, w), device=DEV)
    ray = [r.reshape(1, -1) for r in _rays(s, torch.float32)]
    some = max(1, (6 << 20) // (h * w))
    for a in range(0, F, some):
        T = torch.tensor(Ts[a:a + some], device=DEV, dtype=torch.float32)
        part = scenes[a:a + some]
        d = [T[:, k, 0:1] * ray[0] + T[:, k, 1:2] * ray[1] + T[:, k, 2:3] * ray[2] for k in range(3)]
        o = [T[:, k, 3:4] for k in range(3)]
        inv = [1.0 / torch.where(x == 0, 1e-12, x) for x in d]
        best = torch.full_like(d[0], 1e9)

        def slab(lo_hi, inward):
            t = [((lo_hi[:, k:k + 1] - o[k]) * inv[k], (lo_hi[:, 3 + k:4 + k] - o[k]) * inv[k]) for k in range(3)]
            far = torch.minimum(torch.minimum(torch.maximum(*t[0]), torch.maximum(*t[1])), torch.maximum(*t[2]))
            if inward:
                return far
            near = torch.maximum(torch.maximum(torch.minimum(*t[0]), torch.minimum(*t[1])), torch.minimum(*t[2]))
            return torch.where((near <= far) & (near > 0), near, 1e9)

        def per_frame(key):
            return torch.tensor(np.stack([q[key] for q in part]), device=DEV, dtype=torch.float32)

        if "room" in part[0]:
            best = slab(per_frame("room"), True)
        if "ground" in part[0]:
            t = -o[2] * inv[2]
            best = torch.where(t > 0, t, best)
        boxes = per_frame("boxes")
        for b in range(boxes.shape[1]):
            best = torch.minimum(best, slab(boxes[:, b], False))
        if "balls" in part[0]:
            balls = per_frame("balls")
            dd = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
            for b in range(balls.shape[1]):
                q = [o[k] - balls[:, b, k:k + 1] for k in range(3)]
                qd = q[0] * d[0] + q[1] * d[1] + q[2] * d[2]
                disc = qd * qd - dd * (q[0] ** 2 + q[1] ** 2 + q[2] ** 2 - balls[:, b, 3:4] ** 2)
                t = (-qd - torch.sqrt(torch.clamp(disc, min=0.0))) / dd
                best = torch.where((disc > 0) & (t > 0) & (t < best), t, best)
        noise = torch.randn(best.shape, device=DEV, generator=gen)
        if s["kind"] == "pinhole":
            z = best + 0.0012 * best * best * noise
            lost = torch.rand(best.shape, device=DEV, generator=gen) < 0.05
            z = torch.where(lost | (best > 5.0), 0.0, z)
        else:
            z = torch.where(best < s["max_range"], best + 0.02 * noise, 0.0)
        out[a:a + some] = z.reshape(-1, h, w)
    return out


def _colors(Ts, s, depth, gen):
    """Colour images registered to the depth images: a smooth texture of the world point with a little jitter."""
    out = []
    ray = _rays(s, torch.float32)
    for T, d in zip(Ts, depth):
        x, y, z = ((T[k, 0] * ray[0] + T[k, 1] * ray[1] + T[k, 2] * ray[2]) * d + T[k, 3] for k in range(3))
        tex = torch.stack([128 + 100 * torch.sin(3.1 * x + 1.3 * z), 128 + 100 * torch.sin(2.3 * y - 0.7 * x),
                           128 + 100 * torch.cos(1.7 * z + 2.9 * y)])
        c = (tex + 3 * torch.randn(tex.shape, device=DEV, generator=gen)).clamp(0, 255).to(torch.int32)
        out.append(c[0] | (c[1] << 8) | (c[2] << 16))
    return torch.stack(out)


RIG = [_pinhole(640, 480), _pinhole(640, 480), _pinhole(848, 480), _pinhole(1280, 720)]
SERVE = [_pinhole(320, 240), _pinhole(640, 480), _pinhole(1280, 720), _lidar(1024, 64)]


def _level(T):
    """A LiDAR's pose at a camera's place: z up, x along the camera's heading."""
    L = np.eye(4)
    f = T[:3, 2] * [1, 1, 0]
    L[:3, 0] = f / np.linalg.norm(f)
    L[:3, 2] = [0, 0, 1]
    L[:3, 1] = np.cross(L[:3, 2], L[:3, 0])
    L[:3, 3] = T[:3, 3]
    return L


def _frames(case, seed):
    """The frames of a pass in order: (map, sensor, pose, depth [H, W], colour or None), and each map's voxel size."""
    rs = np.random.RandomState(seed % (1 << 32))
    gen = torch.Generator(device=DEV).manual_seed(seed)
    n, kind = case["frames"], case["kind"]
    if kind in ("rig", "lidar"):
        Ts = _path(rs, n, 20.0, 12.0, 0.15)
        lot = _lot(rs, Ts[:, :3, 3])
        if kind == "lidar":
            s, poses = _lidar(case["width"], case["height"]), np.stack([_level(T) for T in Ts])
            d = _cast([lot] * n, s, poses, gen)
            return [(0, s, poses[i], d[i], None) for i in range(n)], [case["voxel"]]
        sensors, poses = RIG + [_lidar(1024, 64)], []
        for k in range(4):
            c, q = math.cos(k * math.pi / 2), math.sin(k * math.pi / 2)
            R = np.array([[c, -q, 0, 0], [q, c, 0, 0], [0, 0, 1, 0], [0, 0, 0, 1.0]])
            turned = np.stack([R @ np.block([[T[:3, :3], np.zeros((3, 1))], [np.zeros((1, 3)), np.ones((1, 1))]])
                               for T in Ts])
            turned[:, :3, 3] = Ts[:, :3, 3] + 0.1 * turned[:, :3, 2]
            poses.append(turned)
        poses.append(np.stack([_level(T) for T in Ts]))
        d = [_cast([lot] * n, s, P, gen) for s, P in zip(sensors, poses)]
        return [(0, sensors[k], poses[k][i], d[k][i], None) for i in range(n) for k in range(5)], [case["voxel"]]
    if kind == "serve":
        of_case = np.random.RandomState(case["maps"] * 1000 + n)  # the maps and the schedule
        voxels = [(0.02, 0.05, 0.1)[k] for k in of_case.randint(0, 3, case["maps"])]
        paths = [_path(rs, n, 5.0, 2.7, 0.06) for _ in voxels]
        rooms = [_room(rs, P[:, :3, 3]) for P in paths]
        which = [(int(of_case.randint(case["maps"])), int(of_case.randint(4))) for _ in range(n)]
        out = [None] * n
        for k, s in enumerate(SERVE):
            mine = [i for i in range(n) if which[i][1] == k]
            if not mine:
                continue
            P = np.stack([paths[which[i][0]][i] for i in mine])
            P = np.stack([_level(T) for T in P]) if s["kind"] == "lidar" else P
            d = _cast([rooms[which[i][0]] for i in mine], s, P, gen)
            for at, i in enumerate(mine):
                out[i] = (which[i][0], s, P[at], d[at], None)
        return out, voxels
    Ts = _path(rs, n, 5.0, 2.7, 0.06)
    room = _room(rs, Ts[:, :3, 3])
    s = _pinhole(case["width"], case["height"])
    d = _cast([room] * n, s, Ts, gen)
    col = _colors(Ts, s, d, gen) if kind == "color" else [None] * n
    return [(0, s, Ts[i], d[i], col[i]) for i in range(n)], [case["voxel"]]


# ------------------------------------------- the blocks that a frame's band meets

class _Grid:
    """A dense box of block coordinates around everything the frames of one map see."""

    def __init__(self, frames, voxel):
        p = np.stack([T[:3, 3] for _, _, T, _, _ in frames])
        reach = [31.0 if s["kind"] == "lidar" else 7.5 for _, s, _, _, _ in frames]
        lo, hi = (p - np.array(reach)[:, None]).min(0), (p + np.array(reach)[:, None]).max(0)
        lo[2], hi[2] = max(lo[2], -17.0), min(hi[2], 20.0)
        self.lo = np.floor(lo / (8 * voxel)).astype(int) - 1
        self.n = np.floor(hi / (8 * voxel)).astype(int) + 2 - self.lo

    def cells(self):
        return int(self.n.prod())

    def coords(self, at):
        return torch.stack([at // int(self.n[1] * self.n[2]), at // int(self.n[2]) % int(self.n[1]),
                            at % int(self.n[2])], 1) + torch.tensor(self.lo, device=DEV)


def _band(grid, frame, voxel, trunc):
    """Which of the grid's blocks the band segments of a frame's pixels meet (bool per cell, x slowest)."""
    _, s, T, depth, _ = frame
    B, tau = 8 * voxel, _f32(trunc * voxel)
    ok = ((depth > 0) & torch.isfinite(depth)) if s["kind"] == "pinhole" else \
        ((depth >= _f32(s["min_range"])) & (depth <= _f32(s["max_range"])))
    z = depth[ok].double()
    ray = [r[ok] for r in _rays(s, torch.float64)]
    d = [(T[k, 0] * ray[0] + T[k, 1] * ray[1] + T[k, 2] * ray[2]) / B for k in range(3)]
    o = [T[k, 3] / B for k in range(3)]
    s0, s1 = torch.clamp(z - tau, min=0.0), z + tau
    hit = torch.zeros(grid.cells(), dtype=torch.bool, device=DEV)

    def put(cell, take):
        c = [x.long() - int(grid.lo[k]) for k, x in enumerate(cell)]
        for k in range(3):
            take = take & (c[k] >= 0) & (c[k] < int(grid.n[k]))
        at = (c[0] * int(grid.n[1]) + c[1]) * int(grid.n[2]) + c[2]
        hit[at[take]] = True

    first = [torch.floor(o[k] + s0 * d[k]) for k in range(3)]
    put(first, torch.ones_like(z, dtype=torch.bool))
    most = 1 + int(math.ceil(float(torch.stack([x.abs().max() for x in d]).max()) * 2 * tau)) if z.numel() else 0
    for k in range(3):
        up = d[k] > 0
        for q in range(most):
            wall = torch.where(up, first[k] + 1 + q, first[k] - q)
            t = (wall - o[k]) / d[k]
            cell = [torch.floor(o[a] + t * d[a]) for a in range(3)]
            cell[k] = torch.where(up, wall, wall - 1)
            put(cell, (t >= s0) & (t <= s1))
    return hit


def _blocks(frames, voxel, trunc):
    """(grid, the band's cells, (block, frame) pairs) of one map's frames."""
    grid = _Grid(frames, voxel)
    every = torch.zeros(grid.cells(), dtype=torch.int32, device=DEV)
    for f in frames:
        every += _band(grid, f, voxel, trunc)
    return grid, every.nonzero()[:, 0], int(every.sum())


def _centres(grid, at, voxel):
    """float32 centres of the 512 voxels of each block, x fastest."""
    l = torch.arange(512, device=DEV)
    off = torch.stack([l % 8, l // 8 % 8, l // 64], 1)
    g = grid.coords(at)[:, None] * 8 + off[None]
    return ((g.double() + 0.5) * voxel).float().reshape(-1, 3).contiguous()


def _of_map(frames, m):
    return [f for f in frames if f[0] == m]


_counted = {}


def _counts(case):
    """Blocks, (block, frame) pairs and pixels of a pass on the inputs of seed 0: they size the buffers for any seed."""
    key = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    if key not in _counted:
        frames, voxels = _frames(case, 0)
        blocks = pairs = 0
        for m, v in enumerate(voxels):
            mine = _of_map(frames, m)
            if mine:
                _, at, n = _blocks(mine, _f32(v), case["trunc"])
                blocks, pairs = blocks + len(at), pairs + n
        _counted[key] = blocks, pairs, sum(f[3].numel() for f in frames)
    return _counted[key]


def _room_for(case):
    """Blocks that a case's read-out has room for: half as many again as seed 0 has."""
    return _counts(case)[0] * 3 // 2 + 16


# ------------------------------------------------------------------ a pass


def prepare(case, seed):
    kind, trunc, st = case["kind"], case["trunc"], STORAGE[case["storage"]]
    frames, voxels = _frames(case, seed)
    layer = {"occupancy": gt.LAYER_OCCUPANCY, "color": gt.LAYER_COLOR}.get(kind, gt.LAYER_TSDF)
    small = {"max_blocks": 1 << 16} if kind in ("esdf", "serve") else {}
    maps = [gt.TsdfMap(v, trunc, MAX_WEIGHT, storage=st, layer=layer, weighting=case.get("weighting", 0), **small)
            for v in voxels]
    s = {"case": dict(case), "maps": maps, "frames": frames, "reads": []}
    if kind != "mesh":
        # one buffer for the values of all maps, with room to spare
        room = 512 * _room_for(case)
        s["dist"] = torch.zeros((room, 3) if kind == "color" else room, device=DEV)
        s["weight"] = torch.zeros(room, device=DEV)
        a = 0
        for m, v in enumerate(voxels):
            mine = _of_map(frames, m)
            if mine:
                grid, at, _ = _blocks(mine, _f32(v), trunc)
                pts = _centres(grid, at[:(room - a) // 512], _f32(v))
                b = a + len(pts)
                s["reads"].append((maps[m], pts, s["dist"][a:b], s["weight"][a:b]))
                a = b
    if kind == "host":
        h, w = _shape(frames[0][1])
        host = torch.empty((len(frames), h, w), dtype=torch.float32, pin_memory=True)
        for i, f in enumerate(frames):
            host[i].copy_(f[3])
        s["host"] = host
        s["descs"] = [gt.frame_desc_host(0, f[1], f[2], host[i]) for i, f in enumerate(frames)]
        s["staging"] = torch.empty(4 * 32 * ((4 * h * w + 255) // 256 * 256), dtype=torch.uint8, device=DEV)
    elif kind not in ("live", "occupancy", "lidar"):
        s["descs"] = [gt.frame_desc(f[0], f[1], f[2], f[3], f[4]) for f in frames]
    if kind == "mesh":
        gt.integrate_batch([maps[0].handle], s["descs"])
        n = 90 * _room_for(case)  # triangles
        s["out"] = {"pos": torch.zeros((n, 3, 3), device=DEV),
                    "keys": torch.zeros((n, 3, 4), dtype=torch.int32, device=DEV),
                    "cube": torch.zeros((n, 3), dtype=torch.int32, device=DEV)}
    return s


def _batch(s, a, b):
    gt.integrate_batch([m.handle for m in s["maps"]], s["descs"][a:b])


def run(s):
    case, maps, frames = s["case"], s["maps"], s["frames"]
    kind = case["kind"]
    if kind == "mesh":
        if case["changed"]:
            _batch(s, max(0, len(frames) - 8), len(frames))
        out = s["out"]
        pos, keys, cube = maps[0].mesh(changed_only=case["changed"], cap=len(out["pos"]))
        # triangles come in no fixed order: sorted by their cube (a room's voxels fit 10 bits an axis)
        n = len(pos)
        order = torch.sort((cube[:, 2] << 20) + (cube[:, 1] << 10) + cube[:, 0], stable=True)[1][:, None]
        for name, v, k in (("pos", pos, 9), ("keys", keys, 12), ("cube", cube, 3)):
            torch.gather(v.view(n, k), 0, order.expand(n, k), out=out[name][:n].view(n, k))
        return out
    if kind in ("live", "lidar"):
        for _, sensor, T, depth, _ in frames:
            maps[0].integrate(sensor, T, depth)
    elif kind == "occupancy":
        for _, sensor, T, depth, _ in frames:
            maps[0].integrate(sensor, T, depth)
            maps[0].decay(0.05, 0.02)
    else:
        for m in maps:
            m.reset()
        if kind == "host":
            gt.integrate_batch_host([maps[0].handle], s["descs"], s["staging"])
        elif kind == "rig":
            for a in range(0, len(frames), 5):
                _batch(s, a, a + 5)
        elif kind == "serve":
            for a in range(0, len(frames), 32):
                _batch(s, a, a + 32)
        elif kind == "esdf":
            _batch(s, 0, case["first"])
            maps[0].esdf_update()
            _batch(s, case["first"], len(frames))
            maps[0].esdf_update()
            _, pts, dist, _ = s["reads"][0]
            maps[0].esdf_query(pts, dist)
            return {"esdf": s["dist"]}
        else:
            _batch(s, 0, len(frames))
    for m, pts, dist, weight in s["reads"]:
        if kind == "color":
            m.query_color(pts, dist, weight)
        else:
            m.query(pts, dist, weight)
    return {"dist": s["dist"], "weight": s["weight"]}


# ------------------------------------------------------------------ in 64 bits

def _sample(frame, p, guard):
    """Per voxel centre p ([n, 3] in the sensor's frame): voxel depth, sampled depth, whether there is one, pixel."""
    _, s, _, depth, _ = frame
    h, w = _shape(s)
    x, y, z = p.unbind(1)
    if s["kind"] == "pinhole":
        ok = z > 0
        zz = torch.where(ok, z, 1.0)
        u = torch.floor(_f32(s["fu"]) * x / zz + _f32(s["cu"]) + 0.5)
        v = torch.floor(_f32(s["fv"]) * y / zz + _f32(s["cv"]) + 0.5)
        ok = ok & (u >= 0) & (u < w) & (v >= 0) & (v < h)
        at = torch.where(ok, v * w + u, 0.0).long()
        d = depth.reshape(-1)[at].double()
        return z, d, ok & (d > 0) & torch.isfinite(d), at
    r = torch.sqrt(x * x + y * y + z * z)
    u = (torch.atan2(y, x) - _f32(s["theta_start"])) * _f32(w / (2 * math.pi)) - 0.5
    v = (torch.atan2(torch.sqrt(x * x + y * y), z) - _f32(s["phi_start"])) * _f32(h / _f32(s["el_fov"])) - 0.5
    k, j = torch.floor(u), torch.floor(v)
    ok = (r > 0) & (j >= 0) & (j <= h - 2)
    k0, j0 = k.long() % w, torch.where(ok, j, 0.0).long()
    k1 = (k0 + 1) % w
    flat = depth.reshape(-1).double()
    q = [flat[j0 * w + k0], flat[j0 * w + k1], flat[(j0 + 1) * w + k0], flat[(j0 + 1) * w + k1]]
    for a in q:
        ok = ok & (a >= _f32(s["min_range"])) & (a <= _f32(s["max_range"]))
    ok = ok & (torch.stack(q).max(0)[0] - torch.stack(q).min(0)[0] <= guard)
    top, bot = q[0] + (u - k) * (q[1] - q[0]), q[2] + (u - k) * (q[3] - q[2])
    return r, top + (v - j) * (bot - top), ok, None


def _fused(case, frames, voxel):
    """Distance (log-odds, colour) and weight of every voxel of the band's blocks after one pass over the frames."""
    kind, trunc = case["kind"], case["trunc"]
    voxel = _f32(voxel)
    tau = _f32(trunc * voxel)
    grid, at, _ = _blocks(frames, voxel, trunc)
    l = torch.arange(512, device=DEV)
    off = torch.stack([l % 8, l // 8 % 8, l // 64], 1)
    coords = grid.coords(at)
    D = torch.zeros((len(at), 512) + ((3,) if kind == "color" else ()), dtype=torch.float64, device=DEV)
    W = torch.zeros((len(at), 512), dtype=torch.float64, device=DEV)
    wf = case.get("weighting", 0)
    for f in frames:
        T = torch.tensor(f[2], device=DEV)
        mine = _band(grid, f, voxel, trunc)[at].nonzero()[:, 0]
        p = ((coords[mine][:, None] * 8 + off[None]).double() + 0.5) * voxel - T[:3, 3]
        dv, d, ok, pix = _sample(f, (p @ T[:3, :3]).reshape(-1, 3), tau)
        dp = d - dv
        ok = ok & (dp >= -tau)
        if kind == "color":
            ok = ok & (dp <= tau)
            c = f[4].reshape(-1)[pix].long()
            new = torch.stack([c & 255, (c >> 8) & 255, (c >> 16) & 255], 1).double()
            d0, w0 = D[mine].reshape(-1, 3), W[mine].reshape(-1)
            d1 = torch.where(ok[:, None], d0 + (new - d0) / (w0 + 1)[:, None], d0)
            D[mine] = d1.reshape(-1, 512, 3)
            W[mine] = torch.where(ok, torch.clamp(w0 + 1, max=MAX_WEIGHT), w0).reshape(-1, 512)
            continue
        d0, w0 = D[mine].reshape(-1), W[mine].reshape(-1)
        if kind == "occupancy":
            D[mine] = torch.where(ok, d0 + torch.where(dp > 0, _f32(-0.4), _f32(0.85)), d0).reshape(-1, 512)
            D = torch.where(D > 0, torch.clamp(D - _f32(0.05), min=0.0),
                            torch.where(D < 0, torch.clamp(D + _f32(0.02), max=0.0), D))
            continue
        w = torch.ones_like(dp)
        if wf & 1:
            w = w / (dv * dv)
        if wf & 2:
            w = torch.where(dp < -voxel, w * (tau + dp) / (tau - voxel), w)
        ok = ok & (w0 + w > 0)
        d1 = torch.where(ok, d0 + w * (torch.clamp(dp, max=tau) - d0) / torch.where(ok, w0 + w, 1.0), d0)
        D[mine] = d1.reshape(-1, 512)
        W[mine] = torch.where(ok, torch.clamp(w0 + w, max=MAX_WEIGHT), w0).reshape(-1, 512)
    return D.reshape(-1, 3) if kind == "color" else D.reshape(-1), W.reshape(-1)


def exact(case, seed):
    # the distance layer is what its propagation rules find and the mesh what its
    # case table joins: neither has a value apart from those rules
    if case["kind"] in ("esdf", "mesh"):
        return None
    frames, voxels = _frames(case, seed)
    room = 512 * _room_for(case)
    dist = torch.zeros((room, 3) if case["kind"] == "color" else room, dtype=torch.float64, device=DEV)
    weight = torch.zeros(room, dtype=torch.float64, device=DEV)
    a = 0
    for m, v in enumerate(voxels):
        mine = _of_map(frames, m)
        if mine:
            d, w = _fused(case, mine, v)
            b = min(room, a + len(d))
            dist[a:b], weight[a:b] = d[:b - a], w[:b - a]
            a = b
    return {"dist": dist, "weight": weight}


def work(case):
    """Images read, the band's voxels written (and read where the map is not new), points in and values out; per pixel
    the segment's set-up and cells, per voxel of a frame's band the projection and update."""
    blocks, pairs, pixels = _counts(case)
    kind = case["kind"]
    vox = 16 if kind == "color" else 4 if kind == "occupancy" or case["storage"] != "fp32" else 8
    if kind == "mesh":
        # about sixty triangles to a block of the surface: positions, keys and cube of each
        return {"bytes": blocks * 512 * vox + blocks * 60 * 96, "flops": blocks * 512 * 10}
    out = 4 if kind == "esdf" else 16 if kind == "color" else 8
    again = 2 if kind in ("live", "lidar", "occupancy") else 1
    got = {"bytes": pixels * (8 if kind == "color" else 4) + blocks * 512 * (again * vox + vox + 12 + out),
           "flops": pixels * 70 + pairs * 512 * 32}
    if kind == "esdf":
        got["bytes"] += blocks * 512 * 4 * 3
    return got
