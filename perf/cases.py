"""The workloads that performance is measured on: what a user of the voxel map, the batched plane fit and the
multi-stream server has them do, through their public entry points.

Three kinds of case:

``map``    one sensor frame into an accumulated map and a segmentation of it (``VoxelMap``): the robot's own loop.
           The map already holds frames from along the path, so the segmentation covers a grown map.
``fit``    RANSAC, refit and hulls of caller-formed clusters (``fit_planes`` or a ``FitPlan``).
``serve``  a frame from each of many sensor streams through one ``Server``, all results polled.

Scenes (floor, open-tread stair, desk, ramp, boxes, slabs), sensor noise, cluster sizes and outliers are drawn from
the seed; frames are ray-cast on the GPU against convex polyhedra."""
import math

import numpy as np
import torch

from paper_2510_01592_gb300 import serve, vm

DEV = "cuda"


def listed():
    return [
        # the smallest call: a local map of one stair, one sparse scan a step, launch-bound
        dict(name="frame_20k", kind="map", scene="stair", ex=1.0, ey=1.0, ez=0.5, voxel=0.02, sensor="cloud",
             points=20000, before=0, clear=False, window=False, host=False, hyp=64, rounds=1, steppable=True),
        # the headline loop: a depth camera at 640 x 480 over a 4 x 4 x 2 m map at 0.01 m, frames on the device
        dict(name="walk", kind="map", scene="stair", ex=4.0, ey=4.0, ez=2.0, voxel=0.01, sensor="camera", width=640,
             height=480, before=60, clear=False, window=False, host=False, hyp=100, rounds=1, steppable=True),
        # the same loop where the scene moves: the voxels on the frame's rays are cleared first (Eq. 2)
        dict(name="walk_clear", kind="map", scene="stair", ex=4.0, ey=4.0, ez=2.0, voxel=0.01, sensor="camera",
             width=640, height=480, before=60, clear=True, window=False, host=False, hyp=100, rounds=1, steppable=True),
        # the robot-centric 5 x 5 x 5 m window, re-centred before each frame, frames from pinned host memory
        dict(name="walk_window", kind="map", scene="stair", ex=5.0, ey=5.0, ez=5.0, voxel=0.01, sensor="camera",
             width=640, height=480, before=40, clear=False, window=True, host=True, hyp=100, rounds=1, steppable=True),
        # every surface clustered, not only the steppable ones, and up to three planes taken from each cluster
        dict(name="walk_planes3", kind="map", scene="stair", ex=4.0, ey=4.0, ez=2.0, voxel=0.01, sensor="camera",
             width=640, height=480, before=60, clear=False, window=False, host=False, hyp=100, rounds=3,
             steppable=False),
        # a coarse, wide map from a small odd-sized camera image
        dict(name="coarse", kind="map", scene="stair", ex=5.35, ey=3.85, ez=2.0, voxel=0.05, sensor="camera", width=423,
             height=241, before=30, clear=False, window=False, host=False, hyp=100, rounds=1, steppable=True),
        # the largest frame and map: a 128-beam spinning LiDAR, 1.3 M rays, 8 x 8 x 3 m at 0.01 m
        dict(name="lidar", kind="map", scene="clutter", ex=8.0, ey=8.0, ez=3.0, voxel=0.01, sensor="lidar", beams=128,
             steps=10160, before=10, clear=False, window=False, host=False, hyp=100, rounds=1, steppable=True),
        # sixteen robots served by one GPU: extents and resolutions differ, a frame of each a pass
        dict(name="serve_16", kind="serve", streams=16, width=640, height=480, before=10, hyp=100),
        # the smallest fit: one cluster by a direct call
        dict(name="fit_1", kind="fit", clusters=1, lo=10000, hi=30000, hyp=100, outliers=0.1, plan=False),
        # the cluster-parallel ablation's largest point: 16 clusters by a direct call
        dict(name="fit_16", kind="fit", clusters=16, lo=10000, hi=30000, hyp=100, outliers=0.1, plan=False),
        # a frame's worth of clusters from many maps at once, uneven by a factor of 4000, through a reusable plan
        dict(name="fit_2000", kind="fit", clusters=2000, lo=50, hi=200000, hyp=256, outliers=0.05, plan=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["cloud", "camera", "camera", "lidar", "serve", "fit", "fit"])
    if kind == "serve":
        return dict(kind="serve", streams=rng.randint(2, 16), width=rng.randint(160, 640), height=rng.randint(120, 480),
                    before=rng.randint(4, 10), hyp=rng.randint(32, 128))
    if kind == "fit":
        lo = _log(rng, 50, 2000)
        return dict(kind="fit", clusters=_log(rng, 1, 1500), lo=lo, hi=_log(rng, 2 * lo, 150000), hyp=_log(rng, 16, 256),
                    outliers=round(rng.uniform(0.0, 0.2), 3), plan=rng.random() < 0.5)
    c = dict(kind="map", scene="stair", clear=False, window=False, host=rng.random() < 0.3, hyp=_log(rng, 32, 256),
             rounds=1, steppable=True)
    if kind == "cloud":
        c.update(ex=round(rng.uniform(0.6, 2.0), 2), ey=round(rng.uniform(0.6, 2.0), 2), ez=0.5,
                 voxel=rng.choice([0.01, 0.02]), sensor="cloud", points=_log(rng, 2000, 100000), before=0)
    elif kind == "camera":
        c.update(ex=round(rng.uniform(2.0, 6.0), 2), ey=round(rng.uniform(2.0, 6.0), 2), ez=2.0,
                 voxel=rng.choice([0.01, 0.01, 0.02, 0.05]), sensor="camera", width=rng.randint(160, 640),
                 height=rng.randint(120, 480), before=rng.randint(10, 60), clear=rng.random() < 0.3,
                 window=rng.random() < 0.25, rounds=rng.choice([1, 1, 1, 2, 3]), steppable=rng.random() < 0.8)
    else:
        c.update(scene="clutter", ex=round(rng.uniform(4.0, 8.0), 2), ey=round(rng.uniform(4.0, 8.0), 2), ez=3.0,
                 voxel=rng.choice([0.01, 0.02]), sensor="lidar", beams=rng.choice([16, 32, 64, 128]),
                 steps=_log(rng, 1000, 10160), before=rng.randint(4, 10), clear=rng.random() < 0.3)
    return c


# ---------------------------------------------------------------------------------------------------- scenes
# A scene is a float array [prims][6][4] of planes (n, d): a point is inside a primitive when n . x <= d on all six.

def _box(center, half, yaw=0.0, tilt=0.0, az=0.0):
    cy, sy, ca, sa = math.cos(yaw), math.sin(yaw), math.cos(az), math.sin(az)
    k = np.array([[0, 0, ca], [0, 0, sa], [-ca, -sa, 0]])
    rot = (np.eye(3) + math.sin(tilt) * k + (1 - math.cos(tilt)) * k @ k) @ np.array([[cy, -sy, 0], [sy, cy, 0],
                                                                                     [0, 0, 1.0]])
    out = []
    for a in range(3):
        n = rot[:, a]
        out += [np.r_[n, n @ center + half[a]], np.r_[-n, -(n @ center) + half[a]]]
    return np.array(out)


def _slab(lo, hi):
    lo, hi = np.asarray(lo, float), np.asarray(hi, float)
    return _box((lo + hi) / 2, (hi - lo) / 2)


def _stair_scene(rs, ex, ey):
    """Floor, an open-tread stair along +x, a desk, a 15 degree ramp and boxes; also the stair's place."""
    prims = [_slab((-60, -60, -1), (60, 60, 0))]
    steps = int(max(2, min(8, (ex - 0.3) // 0.3)))
    x0, y0, wide = 0.25 * (ex - 0.3 * steps) + rs.uniform(0, 0.1), 0.1 * ey, min(0.8, 0.4 * ey)
    rise = min(0.15, 1.2 / steps)
    for k in range(1, steps + 1):
        prims.append(_slab((x0 + 0.3 * (k - 1), y0, rise * k - 0.03), (x0 + 0.3 * k, y0 + wide, rise * k)))
    if ex >= 2.5:
        dx, dy = rs.uniform(0.4, 0.5) * ex, 0.55 * ey
        prims.append(_slab((dx, dy, 0.69), (dx + 0.3 * ex, dy + 0.2 * ey, 0.72)))
        for lx in (dx, dx + 0.2 * ex):
            prims.append(_slab((lx, dy, 0), (lx + 0.04, dy + 0.04, 0.69)))
    rx, ry, run, s, c = 0.08 * ex, 0.38 * ey, 0.35 * ex, math.sin(math.radians(15)), math.cos(math.radians(15))
    prims.append(np.array([[-s, 0, c, -rx * s], [0, 0, -1, 0], [1, 0, 0, rx + run], [0, -1, 0, -ry],
                           [0, 1, 0, ry + 0.15 * ey], [0, 0, -1, 1.0]]))
    for _ in range(20 if ex >= 2.5 else 4):
        sx, sy, h = *(rs.uniform(0.025, 0.12, 2) * ex), rs.uniform(0.05, 0.4)
        prims.append(_box(np.array([rs.uniform(0.1, 0.9) * ex, rs.uniform(0.78, 0.95) * ey, h / 2]),
                          (sx / 2, sy / 2, h / 2), yaw=rs.uniform(0, 1.5)))
    return np.array(prims), (x0, x0 + 0.3 * steps, y0, y0 + wide, rise)


def _clutter_scene(rs, ex, ey):
    """Two floors and a gallery, open underneath, with 500 tilted boxes and slabs on them."""
    prims = [_slab((-60, -60, -1), (60, 60, 0)), _slab((0, 0.62 * ey, 1.15), (ex, ey, 1.2)),
             _slab((0, 0, 2.15), (0.31 * ex, ey, 2.2))]
    for _ in range(500):
        x, y = rs.uniform(0.1, ex - 0.1), rs.uniform(0.1, ey - 0.1)
        sx, sy, sz = np.exp(rs.uniform(math.log(0.1), math.log(2.0), 3)) * 0.5
        if rs.random() < 1 / 3:
            sz = rs.uniform(0.02, 0.08)
        level = 1.2 if y > 0.62 * ey and rs.random() < 0.5 else 0.0
        if abs(x - ex / 2) < 0.6 + sx and abs(y - ey / 2) < 0.6 + sy:
            continue
        prims.append(_box(np.array([x, y, level + sz / 2]), (sx / 2, sy / 2, sz / 2), rs.uniform(0, 3.1),
                          math.radians(rs.uniform(0, 30)), rs.uniform(0, 6.2)))
    return np.array(prims)


def _cast(prims, origin, dirs, group=4):
    """Distance to the first hit along each direction (inf: none)."""
    n = prims[..., :3]
    num = prims[..., 3] - (n * origin).sum(-1)
    best = torch.full((dirs.shape[0],), math.inf, device=DEV)
    for i in range(0, prims.shape[0], group):
        g = n[i:i + group]
        den = g[..., 0:1] * dirs[:, 0] + g[..., 1:2] * dirs[:, 1] + g[..., 2:3] * dirs[:, 2]
        t = num[i:i + group, :, None] / den
        enter = torch.where(den < 0, t, -math.inf).amax(1)
        leave = torch.where(den > 0, t, math.inf).amin(1)
        out = ((den == 0) & (num[i:i + group, :, None] < 0)).any(1)
        hit = (enter <= leave) & (enter > 0) & ~out
        best = torch.minimum(best, torch.where(hit, enter, math.inf).amin(0))
    return best


def _pose(position, yaw, pitch):
    """Camera axes (x right, y down, z forward) to the map, pitched down."""
    cy, sy, cp, sp = math.cos(yaw), math.sin(yaw), math.cos(pitch), math.sin(pitch)
    rz = np.array([[cy, -sy, 0], [sy, cy, 0], [0, 0, 1.0]])
    ry = np.array([[cp, 0, sp], [0, 1, 0], [-sp, 0, cp]])
    rot = rz @ ry @ np.array([[0, 0, 1.0], [-1, 0, 0], [0, -1, 0]])
    return np.concatenate([rot, np.asarray(position, float)[:, None]], 1)


def _camera_rays(width, height):
    """Directions of an 87 x 58 degree pinhole camera, row-major pixels."""
    u = (torch.arange(width, device=DEV) + 0.5 - width / 2) * (2 * math.tan(math.radians(43.5)) / width)
    v = (torch.arange(height, device=DEV) + 0.5 - height / 2) * (2 * math.tan(math.radians(29.0)) / height)
    d = torch.stack([u.expand(height, width), v[:, None].expand(height, width), torch.ones(height, width, device=DEV)],
                    -1).reshape(-1, 3)
    return d / d.norm(dim=1, keepdim=True)


def _lidar_rays(beams, steps):
    """A spinning LiDAR's directions, beam-major, +-22.5 degrees."""
    el = torch.deg2rad(torch.linspace(-22.5, 22.5, beams, device=DEV))[:, None]
    az = torch.arange(steps, device=DEV)[None] * (2 * math.pi / steps)
    return torch.stack([el.cos() * az.cos(), el.cos() * az.sin(), el.sin().expand(beams, steps)], -1).reshape(-1, 3)


def _frame(gen, prims, rays, pose, near, far, sigma0, sigma1):
    """One frame's points in the sensor's axes, NaN where a ray returns nothing in range."""
    rot = torch.tensor(pose[:, :3], dtype=torch.float32, device=DEV)
    world = rays[:, 0:1] * rot[:, 0] + rays[:, 1:2] * rot[:, 1] + rays[:, 2:3] * rot[:, 2]
    r = _cast(prims, torch.tensor(pose[:, 3], dtype=torch.float32, device=DEV), world)
    noisy = r + torch.randn(r.shape, generator=gen, device=DEV) * (sigma0 + sigma1 * r)
    return torch.where(((r >= near) & (r <= far))[:, None], rays * noisy[:, None], math.nan)


def _walk(stair, ex, ey, s):
    """Camera pose at s in [0, 1] of a walk along the stair, 0.45 m over what is under it."""
    x, y = (0.06 + 0.8 * s) * ex, 0.2 * ey + 0.04 * ey * math.sin(6 * s)
    x0, x1, y0, y1, rise = stair
    z = rise * (int((x - x0) / 0.3) + 1) if x0 <= x < x1 and y0 <= y <= y1 else 0.0
    return _pose((x, y, z + 0.45), 0.35 * math.sin(5 * s), math.radians(25.0))


def _map_frames(case, seed):
    """(frames before, the frames of the passes), each (points, pose)."""
    rs = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    ex, ey = case["ex"], case["ey"]
    ring = 6
    if case["sensor"] == "cloud":  # samples of a stair's surfaces, sigma 3 mm
        out = []
        for _ in range(ring):
            n = case["points"]
            p = torch.rand(n, 3, generator=gen, device=DEV) * torch.tensor([ex, ey, 1.0], device=DEV)
            stair, ramp = p[:, 1] < 0.6 * ey, p[:, 1] > 0.68 * ey
            step = (p[:, 0] / (0.3 * ex)).floor().clamp(max=2) + 1
            z = torch.where(stair, 0.12 * step, torch.where(ramp, p[:, 0] * math.tan(math.radians(10.0)), 0.0))
            riser = stair & (p[:, 2] < 0.25)  # a quarter of the stair's samples fall on its risers
            x = torch.where(riser, (step - 1) * 0.3 * ex, p[:, 0])
            z = torch.where(riser, 0.12 * step - 0.12 * 4 * p[:, 2], z)
            p = torch.stack([x, p[:, 1], z], 1) + 0.003 * torch.randn(n, 3, generator=gen, device=DEV)
            out.append((p.contiguous(), np.eye(4)[:3].astype(np.float32).reshape(12)))
        return [], out
    if case["sensor"] == "camera":
        scene, stair = _stair_scene(rs, ex, ey)
        rays, model = _camera_rays(case["width"], case["height"]), (0.3, 4.0, 0.001, 0.002)
        far = [i / max(1, case["before"] - 1) * 0.9 for i in range(case["before"])]
        poses = [_walk(stair, ex, ey, s) for s in far + [0.9 + 0.0035 * i for i in range(ring)]]
    else:
        scene = _clutter_scene(rs, ex, ey)
        rays, model = _lidar_rays(case["beams"], case["steps"]), (0.5, 20.0, 0.005, 0.0)
        poses = []
        for i in range(case["before"] + ring):
            a = 0.3 * i
            p = np.eye(4)[:3].copy()
            p[:, 3] = (ex / 2 + 0.25 * ex * math.cos(a), ey / 2 + 0.25 * ey * math.sin(a), 0.6)
            poses.append(p)
    prims = torch.tensor(scene, dtype=torch.float32, device=DEV)
    frames = [(_frame(gen, prims, rays, p, *model), p.astype(np.float32).reshape(12)) for p in poses]
    return frames[:case["before"]], frames[case["before"]:]


# ---------------------------------------------------------------------------------------------------- clusters

def _clusters(case, seed):
    """Planar patches on jittered 0.01 m lattices with uniform outliers: points float32 [n, 3], offsets int32 [k + 1].
    Sizes are log-uniform, at the quantiles of the range, so that one case's work is the same for every seed."""
    rs = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    k = case["clusters"]
    q = (rs.permutation(k) + 0.5) / k
    sizes = np.exp(math.log(case["lo"]) + q * math.log(case["hi"] / case["lo"])).astype(np.int64)
    off = np.r_[0, np.cumsum(sizes)]
    tilt, az = np.radians(rs.uniform(0, 35, k)), rs.uniform(0, 2 * math.pi, k)
    n = np.stack([np.sin(tilt) * np.cos(az), np.sin(tilt) * np.sin(az), np.cos(tilt)], 1)
    e1 = np.cross(np.array([1.0, 0, 0]), n)
    e1 /= np.linalg.norm(e1, axis=1, keepdims=True)
    e2 = np.cross(n, e1)
    center = rs.uniform(-8, 8, (k, 3)) * np.array([1, 1, 0.1])
    f32 = dict(dtype=torch.float32, device=DEV)
    cid = torch.repeat_interleave(torch.arange(k, device=DEV), torch.as_tensor(sizes, device=DEV))
    idx = torch.arange(int(off[-1]), device=DEV) - torch.as_tensor(off[:-1], device=DEV)[cid]
    side = torch.as_tensor(np.ceil(np.sqrt(sizes)).astype(np.int64), device=DEV)[cid]
    n_all = idx.numel()
    half = (side - 1).float() / 2
    u = ((idx % side).float() - half) * 0.01 + (torch.rand(n_all, generator=gen, device=DEV) - 0.5) * 0.006
    v = ((idx // side).float() - half) * 0.01 + (torch.rand(n_all, generator=gen, device=DEV) - 0.5) * 0.006
    w = torch.randn(n_all, generator=gen, device=DEV) * 0.001
    c, a, b, m = (torch.tensor(t, **f32)[cid] for t in (center, e1, e2, n))
    p = c + u[:, None] * a + v[:, None] * b + w[:, None] * m
    reach = (half * 0.01 + 0.05)[:, None] * (a.abs() + b.abs()) + 0.05
    stray = (torch.rand(n_all, generator=gen, device=DEV) < case["outliers"])[:, None]
    p = torch.where(stray, c + (torch.rand(n_all, 3, generator=gen, device=DEV) * 2 - 1) * reach, p)
    return p.contiguous(), torch.as_tensor(off.astype(np.int32), device=DEV)


# ---------------------------------------------------------------------------------------------------- the cases

def _streams(case, seed):
    """Extents, resolution and frames of each served stream."""
    rs = np.random.default_rng(seed)
    out = []
    for s in range(case["streams"]):
        ex, ey = (round(float(v), 2) for v in np.random.default_rng(1000 + s).uniform(2.0, 6.0, 2))
        out.append(dict(ex=ex, ey=ey, ez=2.0, voxel=(0.01, 0.02, 0.05)[s % 3], sensor="camera", width=case["width"],
                        height=case["height"], before=case["before"], seed=int(rs.integers(1 << 31))))
    return out


def _dims(c):
    return tuple(int(round(c[a] / c["voxel"])) for a in ("ex", "ey", "ez"))


def prepare(case, seed):
    prm = dict(n_hyp=case["hyp"], seed=seed & 0xFFFF)
    if case["kind"] == "fit":
        xyz, off = _clusters(case, seed)
        prm = vm.segment_params(**prm)
        plan = vm.FitPlan(case["clusters"], xyz.shape[0], prm) if case["plan"] else None
        torch.cuda.synchronize()
        return dict(kind="fit", xyz=xyz, off=off, prm=prm, plan=plan, room=_room(case))
    if case["kind"] == "serve":
        srv = serve.Server(vm.segment_params(**prm), mode="batched", max_batch=16)
        sids, rings = [], []
        for st in _streams(case, seed):
            d = _dims(st)
            bricks = math.prod((v + 7) // 8 for v in d)
            sid = srv.open(d, (0.0, 0.0, -0.05), st["voxel"], brick_capacity=min(bricks, 16384))
            before, ring = _map_frames(st, st["seed"])
            for pts, pose in before:
                srv.submit(sid, pts, pose)
            sids.append(sid)
            rings.append(ring)
        srv.drain()
        while srv.poll(max_results=64, with_planes=False):
            pass
        return dict(kind="serve", srv=srv, sids=sids, rings=rings, i=0,
                    room=_room(dict(kind="map", sensor="camera", rounds=case["streams"])))
    before, ring = _map_frames(case, seed)
    m = vm.VoxelMap(_dims(case), (0.0, 0.0, -0.05), case["voxel"])
    for pts, pose in before:
        m.integrate(pts, pose)
    if case["host"]:
        ring = [(p.cpu().pin_memory(), pose) for p, pose in ring]
    prm = vm.segment_params(classify=1 if case["steppable"] else 0, planes_per_cluster=case["rounds"], **prm)
    if before:  # a running program has segmented its map before
        m.segment(prm)
    return dict(kind="map", map=m, ring=ring, prm=prm, i=0, clear=case["clear"], window=case["window"],
                fresh=case["sensor"] == "cloud", room=_room(case))


# Results come in arrays of one size for all inputs of a case: the records found, then zeros.
PLANE = np.dtype([("normal", np.float32, 3), ("offset", np.float32), ("inlier_count", np.uint32), ("label", np.uint32),
                  ("ransac_normal", np.float32, 3), ("ransac_offset", np.float32), ("basis_u", np.float32, 3),
                  ("basis_v", np.float32, 3), ("hull_origin", np.float32, 3), ("hull_offset", np.uint32),
                  ("hull_count", np.uint32), ("n_points", np.uint32), ("best_h", np.int32), ("flags", np.uint32)])


def _room(case):
    if case["kind"] == "fit":
        planes = case["clusters"]
    else:
        planes = {"camera": 512, "cloud": 512, "lidar": 4096}[case["sensor"]] * case["rounds"]
    return dict(planes=np.zeros(planes, PLANE), xy=np.zeros((planes * 48 + 256, 2), np.int32),
                xyz=np.zeros((planes * 48 + 256, 3), np.float32), n=0, h=0)


def _keep(room, res):
    """The result as arrays of the case's size."""
    n, h = len(res["planes"]), len(res["hull_xy"])
    if n > len(room["planes"]) or h > len(room["xy"]):
        raise RuntimeError("%d planes and %d hull vertices do not fit the room for them" % (n, h))
    room["planes"][:n] = res["planes"]
    room["xy"][:h], room["xyz"][:h] = res["hull_xy"], res["hull_xyz"]
    if n < room["n"]:
        room["planes"][n:room["n"]] = 0
    if h < room["h"]:
        room["xy"][h:room["h"]] = 0
        room["xyz"][h:room["h"]] = 0
    room["n"], room["h"] = n, h
    out = {f: room["planes"][f] for f in PLANE.names}
    out["hull_xy"], out["hull_xyz"], out["count"] = room["xy"], room["xyz"], n
    return out


def run(state):
    if state["kind"] == "fit":
        if state["plan"] is not None:
            return _keep(state["room"], state["plan"].run(state["xyz"], state["off"]))
        return _keep(state["room"], vm.fit_planes(state["xyz"], state["off"], state["prm"]))
    i = state["i"]
    state["i"] = i + 1
    if state["kind"] == "serve":
        srv, got = state["srv"], {}
        for sid, ring in zip(state["sids"], state["rings"]):
            srv.submit(sid, *ring[i % len(ring)])
        while len(got) < len(state["sids"]):
            for r in srv.poll(timeout_ms=1000):
                if r["status"] != vm.VM_OK:
                    raise RuntimeError("a served request failed with status %d" % r["status"])
                got[r["stream"]] = r
        each = [got[s] for s in state["sids"]]
        both = {f: np.concatenate([r[f] for r in each]) for f in ("planes", "hull_xy", "hull_xyz")}
        return dict(_keep(state["room"], both), counts=np.array([len(r["planes"]) for r in each]))
    m = state["map"]
    pts, pose = state["ring"][i % len(state["ring"])]
    if state["fresh"]:
        m.reset()
    if state["window"]:
        m.scroll_to(pose.reshape(3, 4)[:, 3])
    m.integrate(pts, pose, clear=state["clear"])
    return _keep(state["room"], m.segment(state["prm"]))


def work(case):
    """Bytes: a frame's points (12 B), the voxels it touches (28 B of sums and count read and written) and every occupied
    voxel's state read once; a fit reads its points once.  Flops: normals (about 500 a voxel) and the RANSAC tests (6)."""
    if case["kind"] == "fit":
        k, lo, hi = case["clusters"], case["lo"], case["hi"]
        n = k * (hi - lo) / math.log(hi / lo)
        return {"bytes": 12 * n + 4 * k + 700 * k, "flops": 6 * n * case["hyp"]}
    if case["kind"] == "serve":
        each = [work(dict(st, kind="map", hyp=case["hyp"])) for st in _streams(case, 0)]
        return {f: sum(w[f] for w in each) for f in ("bytes", "flops")}
    n = {"cloud": lambda: case["points"], "camera": lambda: case["width"] * case["height"],
         "lidar": lambda: case["beams"] * case["steps"]}[case["sensor"]]()
    occupied = 1.75 * case["ex"] * case["ey"] / case["voxel"] ** 2
    if case["sensor"] == "cloud":
        occupied = min(occupied, n)
    return {"bytes": 12 * n + 56 * min(n, occupied / 4) + 28 * occupied,
            "flops": occupied * (500 + 6 * case["hyp"])}


# ---------------------------------------------------------------------------------------------------- exact values
# Which samples a hypothesis takes and which points count as its inliers is defined in 32 bits (a fused multiply-add
# chain); the planes, offsets, bases and hull points that follow from them are computed here in 64 bits.  A whole map's
# outputs have no such value apart from the program: its labels key the sampling, so that one voxel that is classified
# otherwise changes every number; there the whole numbers (labels, counts, hull vertices) are what is compared.

def _fma(a, b, c):
    """Round-to-nearest 32-bit fused multiply-add of float32 values that are held in float64."""
    return (a * b + c).float().double()


def _distance(n, d, p):
    """|n . p + d| in the 32-bit order of the inlier test: n [..., 3], p [..., 3]."""
    return _fma(n[..., 2], p[..., 2], _fma(n[..., 1], p[..., 1], _fma(n[..., 0], p[..., 0], d))).abs()


def _rn(x):
    return x.float().double()


def _samples(label, hyps, seed, n):
    """Indices [hyps, 3] below n: Philox4x64-10 (Salmon et al. 2011) at counters (label, h, 0, 0), key (seed, 0), each word
    scaled by the high half of its product with n."""
    low = np.uint64(0xFFFFFFFF)
    s32 = np.uint64(32)

    def mul(a, b):  # 64 x 64 bits -> (high, low)
        al, ah, bl, bh = a & low, a >> s32, b & low, b >> s32
        t = al * bl
        u = ah * bl + (t >> s32)
        w = al * bh + (u & low)
        return ah * bh + (u >> s32) + (w >> s32), a * b

    h = np.arange(hyps, dtype=np.uint64)
    x = [np.full(hyps, label, np.uint64), h, np.zeros_like(h), np.zeros_like(h)]
    keys = [np.full(hyps, seed, np.uint64), np.zeros_like(h)]
    m0, m1 = np.full(hyps, 0xD2E7470EE14C6C93, np.uint64), np.full(hyps, 0xCA5A826395121157, np.uint64)
    w0, w1 = np.full(hyps, 0x9E3779B97F4A7C15, np.uint64), np.full(hyps, 0xBB67AE8584CAA73B, np.uint64)
    for _ in range(10):
        (h0, l0), (h1, l1) = mul(m0, x[0]), mul(m1, x[2])
        x = [h1 ^ x[1] ^ keys[0], l1, h0 ^ x[3] ^ keys[1], l0]
        keys = [keys[0] + w0, keys[1] + w1]
    return np.stack([mul(w, np.full(hyps, n, np.uint64))[0] for w in x[:3]], 1).astype(np.int64)


def _hull(x, y):
    """Strict convex hull of integer points, counter-clockwise from the lexicographic minimum."""
    pts = torch.stack([x, y], 1)
    if x.numel() > 256:  # drop what lies strictly inside the polygon through the extremes of 32 directions
        t = torch.arange(32, device=x.device, dtype=torch.float64) * (2 * math.pi / 32)
        best = (x.double() * t.cos()[:, None] + y.double() * t.sin()[:, None]).argmax(1)
        poly = torch.unique_consecutive(pts[best], dim=0)
        e = poly.roll(-1, 0) - poly
        if poly.shape[0] > 2:
            inside = torch.ones(x.numel(), dtype=torch.bool, device=x.device)
            for (ex, ey), (ax, ay) in zip(e.tolist(), poly.tolist()):
                if ex or ey:
                    inside &= ex * (y - ay) - ey * (x - ax) > 0
            pts = pts[~inside]
    pts = sorted(set(map(tuple, pts.tolist())))
    if len(pts) < 3:
        return pts
    def half(seq):
        st = []
        for p in seq:
            while len(st) > 1 and ((st[-1][0] - st[-2][0]) * (p[1] - st[-2][1]) -
                                   (st[-1][1] - st[-2][1]) * (p[0] - st[-2][0])) <= 0:
                st.pop()
            st.append(p)
        return st
    return half(pts)[:-1] + half(pts[::-1])[:-1]


def exact(case, seed):
    if case["kind"] != "fit":
        return None
    xyz, off = _clusters(case, seed)
    H, eps = case["hyp"], float(np.float32(0.01))
    bounds = off.tolist()
    out = {f: [] for f in ("normal", "offset", "ransac_normal", "ransac_offset", "basis_u", "basis_v", "hull_origin",
                           "hull_xyz")}
    for c in range(case["clusters"]):
        p = xyz[bounds[c]:bounds[c + 1]].double()
        n = p.shape[0]
        i = torch.as_tensor(_samples(c, H, seed & 0xFFFF, n), device=DEV)
        distinct = (i[:, 0] != i[:, 1]) & (i[:, 0] != i[:, 2]) & (i[:, 1] != i[:, 2])
        p0, p1, p2 = p[i[:, 0]], p[i[:, 1]], p[i[:, 2]]
        a, b = _rn(p1 - p0), _rn(p2 - p0)
        cross = torch.stack([_fma(a[:, 1], b[:, 2], -_rn(a[:, 2] * b[:, 1])),
                             _fma(a[:, 2], b[:, 0], -_rn(a[:, 0] * b[:, 2])),
                             _fma(a[:, 0], b[:, 1], -_rn(a[:, 1] * b[:, 0]))], 1)
        nn = _fma(cross[:, 2], cross[:, 2], _fma(cross[:, 1], cross[:, 1], _rn(cross[:, 0] * cross[:, 0])))
        ok = distinct & (nn > 0)
        inv = _rn(1.0 / _rn(nn.clamp(min=1e-300).sqrt()))
        m = _rn(cross * inv[:, None])
        d = -_fma(m[:, 2], p0[:, 2], _fma(m[:, 1], p0[:, 1], _rn(m[:, 0] * p0[:, 0])))
        counts = torch.zeros(H, dtype=torch.int64, device=DEV)
        for q in range(0, n, 1 << 18):
            counts += (_distance(m[:, None], d[:, None], p[None, q:q + (1 << 18)]) <= eps).sum(1)
        counts = torch.where(ok, counts, -1).tolist()
        best = max(range(H), key=lambda h: (counts[h], -h))
        if counts[best] < 0:
            return None
        keep = _distance(m[best], d[best], p) <= eps
        t0, t1, t2 = p0[best], p1[best], p2[best]
        rn = torch.linalg.cross(t1 - t0, t2 - t0)
        rn = rn / rn.norm()
        ex = torch.tensor([1.0, 0, 0] if abs(float(m[best][0])) < 0.9 else [0, 1.0, 0], dtype=torch.float64, device=DEV)
        u = torch.linalg.cross(ex, rn)
        u = u / u.norm()
        v = torch.linalg.cross(rn, u)
        inl, o = p[keep], p[0]
        mean = inl.mean(0)
        if inl.shape[0] >= 3:
            w, vec = torch.linalg.eigh((inl - mean).T @ (inl - mean))
            normal = vec[:, 0]
        else:
            normal = rn
        normal = normal if normal[2] >= 0 else -normal
        offset = -(normal @ mean)
        nx, ny, nz = m[best]  # the hull's coordinates are whole numbers of 2^-16 m along the basis as 32 bits have it
        zero = torch.zeros_like(nx)
        uq = torch.stack([zero, -nz, ny] if abs(float(nx)) < 0.9 else [nz, zero, -nx])
        uq = _rn(uq * _rn(1.0 / _rn(_fma(uq[2], uq[2], _fma(uq[1], uq[1], _rn(uq[0] * uq[0]))).sqrt())))
        vq = torch.stack([_fma(ny, uq[2], -_rn(nz * uq[1])), _fma(nz, uq[0], -_rn(nx * uq[2])),
                          _fma(nx, uq[1], -_rn(ny * uq[0]))])
        r = _rn(inl - o)
        x, y = (_rn(_fma(r[:, 2], t[2], _fma(r[:, 1], t[1], _rn(r[:, 0] * t[0]))) * 65536).round().long()
                for t in (uq, vq))
        q = torch.tensor(_hull(x, y), dtype=torch.float64, device=DEV).reshape(-1, 2) / 65536
        xyz_h = o + q[:, :1] * u + q[:, 1:] * v
        xyz_h = xyz_h - (xyz_h @ normal + offset)[:, None] * normal
        for f, val in (("normal", normal), ("offset", offset), ("ransac_normal", rn),
                       ("ransac_offset", -(rn @ t0)), ("basis_u", u), ("basis_v", v), ("hull_origin", o)):
            out[f].append(val)
        out["hull_xyz"].append(xyz_h)
    hull = torch.cat(out.pop("hull_xyz")).cpu().numpy()
    room = _room(case)
    r = dict.fromkeys(PLANE.names + ("hull_xy", "count"))
    r.update({f: torch.stack(x).cpu().numpy() for f, x in out.items()})
    r["hull_xyz"] = np.r_[hull, np.zeros((len(room["xyz"]) - len(hull), 3))]
    return r
