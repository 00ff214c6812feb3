"""Performance cases: the work that users of this framework have it do, through its public calls.

A case is a dict of plain values; prepare() builds a seeded map, scans and poses for it, run()
makes one call, work() counts the bytes and operations that call cannot do without, and exact()
evaluates the same quantities in 64-bit torch without this package. The scenes are of the shapes
that the benchmark and the tests use: cluttered rooms seen by Kinect-like pinhole cameras, and
an outdoor terrain with buildings seen by a panoramic Lidar (a ray table) and by cameras.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1702_06813_gb300 as rm

FO, FU, NAN = 0, 1, 2
EPS = 0.1  # Table I's inlier threshold, metres


def listed():
    return [
        # one evaluation of a small camera against a small map: the latency of a single call, as
        # an interactive tracker or an outer optimiser on the host makes it
        dict(name="cost_grad_one_160x120", op="cost_grad", scene="room", tris=20_000, width=160,
             height=120, n=1),
        # the candidate-pose batch of scan matching: 256 poses of a Kinect scan in a mapped room
        dict(name="cost_grad_256_640x480", op="cost_grad", scene="room", tris=1_000_000, width=640,
             height=480, n=256),
        # the same kind of batch at half resolution as problems of one batched call
        dict(name="cost_grad_batch_256_320x240", op="cost_grad_batch", scene="room",
             tris=1_000_000, width=320, height=240, n=256),
        # candidate poses of a panoramic Lidar scan on an outdoor map
        dict(name="cost_grad_64_lidar_1024x64", op="cost_grad", scene="terrain", tris=2_000_000,
             width=1024, height=64, n=64, sensor="lidar"),
        # point-to-plane ICP terms of candidate poses
        dict(name="icp_terms_64_640x480", op="icp_terms", scene="room", tris=500_000, width=640,
             height=480, n=64, tol=0.1),
        # z-buffers with triangle ids and barycentrics, as map maintenance and viewers take them
        dict(name="render_16_640x480", op="render", scene="room", tris=500_000, width=640,
             height=480, n=16),
        # the backward pass to the map: vertex gradients of a window of poses
        dict(name="vertex_grad_16_640x480", op="vertex_grad", scene="room", tris=500_000,
             width=640, height=480, n=16),
        # normals of recorded depth frames, in batches
        dict(name="normals_64_640x480", op="normals", scene="room", tris=0, width=640, height=480,
             n=64, sigma=1.5, metric=True),
        # one depth frame to a labelled mesh (every frame of sequential mapping)
        dict(name="meshify_640x480", op="meshify", scene="room", tris=0, width=640, height=480,
             n=1, step=1),
        # aligning one depth frame to the map by ICP, host result
        dict(name="icp_align_640x480", op="icp_align", scene="room", tris=500_000, width=640,
             height=480, n=1, tol=0.2),
        # a tracking frame: agents with mixed sensors (two cameras and a Lidar), five LM
        # iterations each, in one call
        dict(name="track_24_mixed", op="track", scene="terrain", tris=2_000_000, width=640,
             height=480, n=24, iters=5),
        # the paper's own optimiser: derivative-free search on the Table I cost
        dict(name="dfo_align_320x240", op="dfo_align", scene="room", tris=20_000, width=320,
             height=240, n=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["cost_grad", "cost_grad", "cost_grad_batch", "lidar", "lidar", "icp_terms",
                     "render", "vertex_grad", "normals", "meshify", "icp_align", "track",
                     "dfo_align"])
    w = _log(rng, 96, 640)
    h = max(48, min(480, int(round(w * rng.uniform(0.55, 0.85)))))
    tris = _log(rng, 10_000, 1_000_000)
    if op == "lidar":
        return dict(op="cost_grad", scene="terrain", sensor="lidar", tris=_log(rng, 60_000, 2_000_000),
                    width=_log(rng, 180, 1024), height=_log(rng, 16, 64), n=_log(rng, 1, 64))
    if op in ("cost_grad", "cost_grad_batch"):
        return dict(op=op, scene="room", tris=tris, width=w, height=h, n=_log(rng, 1, 256))
    if op == "icp_terms":
        return dict(op=op, scene="room", tris=tris, width=w, height=h, n=_log(rng, 1, 128),
                    tol=round(rng.uniform(0.05, 0.3), 3))
    if op in ("render", "vertex_grad"):
        return dict(op=op, scene="room", tris=tris, width=w, height=h, n=_log(rng, 1, 16))
    if op == "normals":
        return dict(op=op, scene="room", tris=0, width=w, height=h, n=_log(rng, 1, 64),
                    sigma=round(rng.choice([0.0, rng.uniform(0.5, 4.0)]), 2), metric=rng.random() < 0.5)
    if op == "meshify":
        return dict(op=op, scene="room", tris=0, width=w, height=h, n=1, step=rng.choice([1, 2, 3]))
    if op == "icp_align":
        return dict(op=op, scene="room", tris=tris, width=w, height=h, n=1, tol=round(rng.uniform(0.1, 0.3), 3))
    if op == "track":
        return dict(op=op, scene="terrain", tris=_log(rng, 60_000, 1_500_000), width=w, height=h,
                    n=_log(rng, 2, 24), iters=rng.randint(2, 5))
    return dict(op=op, scene="room", tris=min(tris, 200_000), width=min(w, 320), height=min(h, 240), n=1)


# ---------------------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------------------

_BODY_CAM = np.array([[0.0, 0.0, 1.0], [-1.0, 0.0, 0.0], [0.0, -1.0, 0.0]])


def _rot(v):
    """Rotation matrix of a rotation vector."""
    t = float(np.linalg.norm(v))
    if t < 1e-12:
        return np.eye(3)
    k = np.array([[0, -v[2], v[1]], [v[2], 0, -v[0]], [-v[1], v[0], 0]]) / t
    return np.eye(3) + math.sin(t) * k + (1.0 - math.cos(t)) * (k @ k)


def _pose(position, yaw, pitch=0.0, roll=0.0):
    """Camera-to-world pose of a body with x forward, y left, z up."""
    r = _rot([0, 0, yaw]) @ _rot([0, pitch, 0]) @ _rot([roll, 0, 0])
    t = np.eye(4)
    t[:3, :3] = r @ _BODY_CAM
    t[:3, 3] = position
    return t


def _moved(pose, r, sigma_m, sigma_deg):
    """A pose drawn around `pose` (camera-frame displacement, normal on each axis)."""
    d = np.eye(4)
    d[:3, :3] = _rot(r.normal(scale=math.radians(sigma_deg), size=3))
    d[:3, 3] = r.normal(scale=sigma_m, size=3)
    return pose @ d


def _box_rects(lo, hi, sides=range(6)):
    dx, dy, dz = hi - lo
    x, y, z = np.array([dx, 0, 0.0]), np.array([0, dy, 0.0]), np.array([0, 0, dz])
    all6 = [(lo, y, x), (lo + z, x, y), (lo, x, z), (lo + y, z, x), (lo, z, y), (lo + x, y, z)]
    return [all6[s] for s in sides]


def _grid(rects, target, label):
    """Rectangles (origin, edge, edge) as grids of about `target` triangles in all."""
    if not rects or target <= 0:
        return np.zeros((0, 3), np.float32), np.zeros((0, 3), np.int32), np.zeros(0, np.uint8)
    e = np.array([(np.linalg.norm(u), np.linalg.norm(v)) for _, u, v in rects])
    lo, hi = 1e-4, 100.0
    for _ in range(60):
        mid = math.sqrt(lo * hi)
        n = np.maximum(1, np.ceil(e / mid))
        lo, hi = (mid, hi) if 2 * np.sum(n[:, 0] * n[:, 1]) > target else (lo, mid)
    vs, fs, base = [], [], 0
    for (o, u, v), (nu, nv) in zip(rects, np.maximum(1, np.ceil(e / hi)).astype(int)):
        a, b = np.meshgrid(np.arange(nu + 1) / nu, np.arange(nv + 1) / nv, indexing="ij")
        vs.append((o + a[..., None] * u + b[..., None] * v).reshape(-1, 3).astype(np.float32))
        i, j = np.meshgrid(np.arange(nu), np.arange(nv), indexing="ij")
        q = (i * (nv + 1) + j).ravel() + base
        fs.append(np.stack([q, q + nv + 1, q + nv + 2, q, q + nv + 2, q + 1], 1).reshape(-1, 3).astype(np.int32))
        base += (nu + 1) * (nv + 1)
    f = np.concatenate(fs)
    return np.concatenate(vs), f, np.full(len(f), label, np.uint8)


def _panels(r, fixed, places, n, size, off):
    """Free-unknown panels standing off the sides of the places (lo, hi; sign +1: outside)."""
    rects = []
    for _ in range(n):
        lo, hi, sign = places[r.integers(len(places))]
        w, h = fixed.uniform(*size), fixed.uniform(*size)
        d, side = r.uniform(*off) * sign, r.integers(4)
        z = r.uniform(lo[2] + 0.1, max(lo[2] + 0.2, hi[2] - h - 0.1))
        ax = 0 if side < 2 else 1
        s = r.uniform(lo[ax], max(lo[ax] + 0.01, hi[ax] - w))
        c = lo[1 - ax] - d if side % 2 == 0 else hi[1 - ax] + d
        o = np.array([s, c, z]) if ax == 0 else np.array([c, s, z])
        u = np.array([w, 0, 0.0]) if ax == 0 else np.array([0, w, 0.0])
        rects.append((o, u, np.array([0, 0, h])))
    return rects


def _join(parts):
    v, f, lab, base = [], [], [], 0
    for pv, pf, pl in parts:
        v.append(pv)
        f.append(pf + np.int32(base))
        lab.append(pl)
        base += len(pv)
    return (np.ascontiguousarray(np.concatenate(v)), np.ascontiguousarray(np.concatenate(f)), np.concatenate(lab))


def _free(p, boxes, margin):
    return not any(np.all(p > lo - margin) and np.all(p < hi + margin) for lo, hi in boxes)


def _fixed(tris):
    """Sizes of things, the same for every seed: so are then the numbers of vertices and faces."""
    return np.random.Generator(np.random.PCG64(tris))


def _room(r, tris):
    """A 10 x 8 x 3 m room with clutter; a fifth of the triangles are frontier panels. Small maps
    are a 5 x 4 x 3 m room."""
    fixed = _fixed(tris)
    big = tris == 0 or tris > 100_000
    size = np.array([10.0, 8.0, 3.0] if big else [5.0, 4.0, 3.0])
    lo, hi = -size / 2 * [1, 1, 0], size / 2 * [1, 1, 0] + [0, 0, size[2]]
    boxes = []
    for _ in range(120 if big else 30):
        d = fixed.uniform(0.2, 1.0, 3)
        p = np.array([r.uniform(lo[0], hi[0] - d[0]), r.uniform(lo[1], hi[1] - d[1]), 0.0])
        boxes.append((p, p + d))
    scene = dict(kind="room", boxes=boxes, room=(lo, hi))
    if tris:
        rects = _box_rects(lo, hi) + [q for b in boxes for q in _box_rects(*b)]
        panels = _panels(r, fixed, [(lo, hi, -1.0)], 40, (0.3, 1.0), (0.2, 0.5)) if big else []
        n_fu = tris // 5 if panels else 0
        scene["mesh"] = _join([_grid(rects, tris - n_fu, FO), _grid(panels, n_fu, FU)])
    return scene


def _room_pose(r, scene):
    lo, hi = scene["room"]
    for _ in range(1000):
        p = np.array([r.uniform(lo[0] + 0.7, hi[0] - 0.7), r.uniform(lo[1] + 0.7, hi[1] - 0.7), r.uniform(1.1, 2.0)])
        if _free(p, scene["boxes"], 0.75):
            break
    return _pose(p, r.uniform(-math.pi, math.pi), r.uniform(-0.17, 0.17), r.uniform(-0.17, 0.17))


def _height(waves, x, y):
    h = 0.0
    for a, kx, ky, ph in waves:
        h = h + a * (torch.sin(kx * x + ky * y + ph) if torch.is_tensor(x) else np.sin(kx * x + ky * y + ph))
    return h


def _terrain(r, tris):
    """A 200 x 200 m rolling terrain with 40 buildings; three tenths of the triangles are
    frontier panels around the buildings."""
    half, fixed = 100.0, _fixed(tris)
    waves = []
    for o in range(6):
        f, th = 2 * math.pi * 2 ** o / 60.0, r.uniform(0, 2 * math.pi)
        waves.append((1.6 / 2 ** o, f * math.cos(th), f * math.sin(th), r.uniform(0, 2 * math.pi)))
    boxes = []
    for _ in range(40):
        d = np.array([fixed.uniform(5, 30), fixed.uniform(5, 30), fixed.uniform(5, 22)])
        p = np.array([r.uniform(-98, 98 - d[0]), r.uniform(-98, 98 - d[1]), 0.0])
        p[2] = float(_height(waves, p[0] + d[0] / 2, p[1] + d[1] / 2)) - 2.0
        boxes.append((p, p + d))
    scene = dict(kind="terrain", boxes=boxes, waves=waves, half=half)
    n_fu = int(0.3 * tris)
    walls = [q for b in boxes for q in _box_rects(*b, sides=range(1, 6))]
    area = sum(np.linalg.norm(u) * np.linalg.norm(v) for _, u, v in walls)
    n_walls = int((tris - n_fu) * area / (area + 4 * half * half))
    n = max(2, int(round(math.sqrt((tris - n_fu - n_walls) / 2))))
    ground = _grid([(np.array([-half, -half, 0.0]), np.array([2 * half, 0, 0.0]), np.array([0, 2 * half, 0.0]))],
                   2 * n * n, FO)
    ground[0][:, 2] = _height(waves, ground[0][:, 0].astype(np.float64), ground[0][:, 1].astype(np.float64))
    panels = _panels(r, fixed, [(lo, hi, 1.0) for lo, hi in boxes], 400, (2.0, 8.0), (1.0, 5.0))
    scene["mesh"] = _join([ground, _grid(walls, n_walls, FO), _grid(panels, n_fu, FU)])
    return scene


def _terrain_pose(r, scene, lift, pitch=0.0):
    for _ in range(1000):
        x, y = r.uniform(-60, 60, 2)
        p = np.array([x, y, float(_height(scene["waves"], x, y)) + lift])
        if _free(p, scene["boxes"], 3.0):
            break
    return _pose(p, r.uniform(-math.pi, math.pi), pitch)


def _pinhole(w, h, near, far_range):
    f = 525.0 * w / 640.0
    return dict(model="pinhole", width=w, height=h, fx=f, fy=f, cx=w / 2.0, cy=h / 2.0, near=near,
                range_min=near, range_max=far_range)


def _lidar(w, h):
    return dict(model="lidar", width=w, height=h, az0=-math.pi, az_step=2 * math.pi / w, el0=math.radians(15.0),
                el_step=math.radians(40.0) / max(h - 1, 1), near=1.0, range_min=1.0, range_max=80.0)


def _rays(cam):
    """(H, W, 3) float64 rays on the GPU (z = 1 for a pinhole, unit for the Lidar)."""
    j, i = torch.meshgrid(torch.arange(cam["height"], dtype=torch.float64, device="cuda"),
                          torch.arange(cam["width"], dtype=torch.float64, device="cuda"), indexing="ij")
    if cam["model"] == "pinhole":
        return torch.stack([(i + 0.5 - cam["cx"]) / cam["fx"], (j + 0.5 - cam["cy"]) / cam["fy"], torch.ones_like(i)], -1)
    az, el = cam["az0"] + cam["az_step"] * (i + 0.5), cam["el0"] - cam["el_step"] * j
    return torch.stack([torch.cos(el) * torch.sin(az), -torch.sin(el), torch.cos(el) * torch.cos(az)], -1)


def _cast(scene, cam, pose):
    """Distance along each ray to the world's solids (inf: none), (H, W) float64."""
    P = torch.as_tensor(pose, device="cuda")
    o, d = P[:3, 3], (_rays(cam) @ P[:3, :3].T).reshape(-1, 3)
    inv = 1.0 / d
    best = torch.full((d.shape[0],), math.inf, dtype=torch.float64, device="cuda")
    for lo, hi in scene["boxes"]:
        a = (torch.as_tensor(lo, device="cuda") - o) * inv
        b = (torch.as_tensor(hi, device="cuda") - o) * inv
        t0, t1 = torch.minimum(a, b).amax(1), torch.maximum(a, b).amin(1)
        best = torch.where((t1 >= t0) & (t0 > 0) & (t0 < best), t0, best)
    if scene["kind"] == "room":
        lo, hi = (torch.as_tensor(x, device="cuda") for x in scene["room"])
        t1 = torch.maximum((lo - o) * inv, (hi - o) * inv).amin(1)
        best = torch.minimum(best, t1)
    else:
        hit = torch.full_like(best, math.inf)
        for k in range(1, 165):  # march, then one secant step inside the first crossing
            t = 0.5 * k
            p = o + t * d
            up = p[:, 2] - _height(scene["waves"], p[:, 0], p[:, 1])
            if k > 1:
                f = was / (was - up)
                hit = torch.where((up <= 0) & (was > 0) & torch.isinf(hit), t - 0.5 + 0.5 * f, hit)
            was = up
        best = torch.minimum(best, hit)
    return best.reshape(cam["height"], cam["width"])


def _observe(scene, cam, pose, r, rel=0.005, absolute=0.0, drop=0.02):
    """Depth and class of one observed range image, with noise and dropout, on the GPU. Depth
    cameras have no values in a band along the right border."""
    t = _cast(scene, cam, pose)
    n = torch.as_tensor(r.standard_normal(t.numel(), dtype=np.float32), device="cuda").reshape(t.shape).double()
    u = torch.as_tensor(r.random(t.numel(), dtype=np.float32), device="cuda").reshape(t.shape)
    t = t + n * (absolute + rel * torch.where(torch.isfinite(t), t, torch.zeros_like(t)))
    none = ~(t <= cam["range_max"]) | (u < drop)
    t = torch.where(none, torch.full_like(t, cam["range_max"]), t)
    dead = ~none & (t < cam["range_min"])
    if cam["model"] == "pinhole":
        dead[:, cam["width"] - cam["width"] // 80:] = True
        none &= ~dead
    cls = none.to(torch.uint8) * FU + dead.to(torch.uint8) * NAN
    return torch.where(dead, torch.full_like(t, math.nan), t).float().contiguous(), cls.contiguous()


def _intr(cam):
    if cam["model"] == "pinhole":
        return rm.Intrinsics(rm.RM_PINHOLE, cam["width"], cam["height"], cam["fx"], cam["fy"], cam["cx"], cam["cy"],
                             near=cam["near"])
    return rm.Intrinsics(rm.RM_RAYTABLE, cam["width"], cam["height"], az0=cam["az0"], az_step=cam["az_step"],
                         el0=cam["el0"], el_step=cam["el_step"], near=cam["near"],
                         rays=_rays(cam).float().contiguous())


def _inputs(case, seed):
    """Everything the call takes, without the framework's objects."""
    r = np.random.Generator(np.random.PCG64([seed, case["width"], case["height"], case["n"], case["tris"]]))
    scene = _room(r, case["tris"]) if case["scene"] == "room" else _terrain(r, case["tris"])
    s = dict(mesh=scene.get("mesh"))
    op, w, h, n = case["op"], case["width"], case["height"], case["n"]
    if op == "track":
        cams = [_pinhole(max(w // 4, 48), max(h // 4, 36), 0.3, 40.0), _pinhole(w, h, 0.3, 40.0), _lidar(1024, 64)]
        s["cams"], s["kinds"], s["scans"], s["poses"] = cams, [k % 3 for k in range(n)], [], []
        for k in s["kinds"]:
            gt = _terrain_pose(r, scene, 1.8 if k == 2 else 1.5, 0.0 if k == 2 else 0.26)
            s["scans"].append(_observe(scene, cams[k], gt, r, *((0.0, 0.02) if k == 2 else (0.005, 0.0))))
            s["poses"].append(_moved(gt, r, 0.02, 0.2))
        return s
    lidar = case.get("sensor") == "lidar"
    cam = _lidar(w, h) if lidar else _pinhole(w, h, 0.5 if w > 200 else 0.1, 4.5 if w > 200 else 4.0)
    s["cam"] = cam
    if op == "normals":
        frames = [_observe(scene, cam, _room_pose(r, scene), r) for _ in range(min(n, 4))]
        s["depth"] = torch.stack([frames[k % len(frames)][0] * (1.0 + 0.01 * (k // len(frames))) for k in range(n)])
        s["cls"] = torch.stack([frames[k % len(frames)][1] for k in range(n)])
        return s
    gt = _terrain_pose(r, scene, 1.8) if lidar else _room_pose(r, scene)
    s["scan"] = _observe(scene, cam, gt, r, *((0.0, 0.02) if lidar else (0.005, 0.0)))
    if op == "meshify":
        s["pose"] = gt
    elif op in ("icp_align", "dfo_align"):
        s["pose"] = _moved(gt, r, 0.03, 1.0)
    elif lidar:
        s["poses"] = np.stack([_moved(gt, r, 0.17, 1.7) for _ in range(n)])
    else:
        s["poses"] = np.stack([_moved(gt, r, 0.10, 5.0) for _ in range(n)])
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    st = dict(case=case, op=case["op"])
    if s["mesh"] is not None:
        st["map"] = rm.Map(*s["mesh"])
    if case["op"] == "track":
        intr = [_intr(c) for c in s["cams"]]
        st["problems"] = [(rm.Scan.make(intr[k], *sc), p) for k, sc, p in zip(s["kinds"], s["scans"], s["poses"])]
        return st
    intr = st["intr"] = _intr(s["cam"])
    if "scan" in s:
        st["scan"] = rm.Scan.make(intr, *s["scan"])
    for k in ("depth", "cls", "pose"):
        if k in s:
            st[k] = s[k]
    if "poses" in s:
        st["poses"] = torch.as_tensor(s["poses"], device="cuda")
    return st


def run(state):
    op, c = state["op"], state["case"]
    if op == "cost_grad":
        return rm.cost_grad(state["map"], state["scan"], state["poses"])
    if op == "cost_grad_batch":
        return rm.cost_grad_batch(state["map"], scans=state["scan"], poses=state["poses"])
    if op == "icp_terms":
        return rm.icp_terms(state["map"], state["scan"], state["poses"], tol=c["tol"])
    if op == "render":
        return rm.render_depth(state["map"], state["poses"], state["intr"], want_id=True, want_bary=True)
    if op == "vertex_grad":
        return rm.cost_grad_vertices(state["map"], state["scan"], state["poses"])
    if op == "normals":
        return rm.depth_normals(state["intr"], state["depth"], state["cls"], sigma=c["sigma"], metric=c["metric"])
    if op == "meshify":
        return rm.meshify(state["scan"], state["pose"], 4.5, step=c["step"])
    if op == "icp_align":
        pose, rep = rm.icp_align(state["map"], state["scan"], state["pose"], tol=c["tol"])
        return {"pose": pose, **{k: v for k, v in rep.items() if k != "status"}}
    if op == "dfo_align":
        pose, rep = rm.dfo_align(state["map"], state["scan"], state["pose"])
        return {"pose": pose, **{k: v for k, v in rep.items() if k != "status"}}
    poses, reps, _ = rm.align_batch(state["map"], state["problems"], max_iters=c["iters"])
    return {"poses": poses, **{k: np.array([r[k] for r in reps]) for k in reps[0]}}


def work(case):
    op, n, px = case["op"], case["n"], case["width"] * case["height"]
    t = case["tris"]
    mesh = 12 * (t // 2) + 13 * t  # about one vertex for two triangles
    if op in ("cost_grad", "cost_grad_batch"):
        rays = 12 * px if case.get("sensor") == "lidar" else 0
        return dict(bytes=mesh + rays + 5 * px + n * (128 + 280), flops=90 * px * n)
    if op == "icp_terms":
        return dict(bytes=mesh + 5 * px + n * (128 + 248), flops=90 * px * n)
    if op == "render":
        return dict(bytes=mesh + n * (128 + 16 * px), flops=40 * px * n)
    if op == "vertex_grad":
        return dict(bytes=mesh + 5 * px + 128 * n + 24 * (t // 2), flops=60 * px * n)
    if op == "normals":
        taps = 2 * math.ceil(3 * case["sigma"]) + 1
        return dict(bytes=17 * px * n, flops=(4 * taps + 20) * px * n)
    if op == "meshify":
        g = ((case["width"] - 1) // case["step"] + 1) * ((case["height"] - 1) // case["step"] + 1)
        return dict(bytes=5 * px + 12 * g + 26 * g, flops=60 * g)
    if op == "icp_align":  # about five evaluations
        return dict(bytes=mesh + 5 * px, flops=5 * 90 * px)
    if op == "dfo_align":  # about 200 scored poses
        return dict(bytes=mesh + 5 * px, flops=200 * 20 * px)
    sizes = [max(case["width"] // 4, 48) * max(case["height"] // 4, 36), px, 1024 * 64]
    total = sum(sizes[k % 3] for k in range(n))
    return dict(bytes=mesh + 5 * total + 12 * 65536, flops=(case["iters"] + 1) * 90 * total)


# ---------------------------------------------------------------------------------------
# the same quantities in 64-bit torch
# ---------------------------------------------------------------------------------------

def _visible(v, f, cam, rays, pose):
    """Triangle per pixel (-1: none), its depth along the pixel's ray and the corners in the
    camera frame of one view, by the exact test of each pixel ray against each triangle whose
    bounding rectangle holds the pixel."""
    W, H, dev = cam["width"], cam["height"], v.device
    P = torch.as_tensor(pose, device=dev)
    c = (v - P[:3, 3]) @ P[:3, :3]
    a = c[f]  # (T, 3 corners, 3)
    if cam["model"] == "pinhole":
        near = cam["near"]
        z = a[..., 2]
        front = z >= near
        b = a.roll(-1, 1)
        s = (near - z) / (b[..., 2] - z)
        cut = a + s[..., None] * (b - a)
        crosses = front != front.roll(-1, 1)
        pts = torch.cat([a, cut], 1)
        use = torch.cat([front, crosses], 1)
        xy = [cam["f" + k] * pts[..., m] / torch.where(use, pts[..., 2], torch.ones_like(pts[..., 2])) + cam["c" + k]
              for m, k in enumerate("xy")]
        lim = [torch.where(use, q, torch.full_like(q, s_)) for q in xy for s_ in (math.inf, -math.inf)]
        i0, i1 = torch.ceil(lim[0].amin(1) - 0.5 - 1e-6), torch.floor(lim[1].amax(1) - 0.5 + 1e-6)
        j0, j1 = torch.ceil(lim[2].amin(1) - 0.5 - 1e-6), torch.floor(lim[3].amax(1) - 0.5 + 1e-6)
        ok = use.any(1)
        wrap = torch.zeros_like(ok)
    else:
        u = a / a.norm(dim=-1, keepdim=True).clamp_min(1e-30)
        az, el = torch.atan2(u[..., 0], u[..., 2]), torch.asin((-u[..., 1]).clamp(-1, 1))
        chord = torch.stack([(u[:, k] - u[:, (k + 1) % 3]).norm(dim=-1) for k in range(3)]).amax(0)
        bulge = 0.6 * chord  # a great-circle edge leaves its end points' band by less
        wide = (u[..., 1].abs().amax(1) > 0.85) & (chord > 0.05)
        span = az.amax(1) - az.amin(1)
        wrap = span > math.pi
        i0 = torch.ceil((az.amin(1) - cam["az0"]) / cam["az_step"] - 0.5 - 0.01)
        i1 = torch.floor((az.amax(1) - cam["az0"]) / cam["az_step"] - 0.5 + 0.01)
        bulge = bulge * chord
        j0 = torch.ceil((cam["el0"] - el.amax(1) - bulge) / cam["el_step"] - 0.01)
        j1 = torch.floor((cam["el0"] - el.amin(1) + bulge) / cam["el_step"] + 0.01)
        every = wrap | wide
        i0, i1 = torch.where(every, torch.zeros_like(i0), i0), torch.where(every, torch.full_like(i1, W - 1), i1)
        j0 = torch.where(wide, torch.zeros_like(j0), j0)
        j1 = torch.where(wide, torch.full_like(j1, H - 1), j1)
        ok = torch.ones_like(wrap)
    i0, i1 = i0.clamp(0, W).nan_to_num(0), i1.clamp(-1, W - 1).nan_to_num(-1)
    j0, j1 = j0.clamp(0, H).nan_to_num(0), j1.clamp(-1, H - 1).nan_to_num(-1)
    count = (i1 - i0 + 1).clamp_min(0) * (j1 - j0 + 1).clamp_min(0) * ok
    tri = torch.nonzero(count > 0).squeeze(1)
    cnt = count[tri].long()
    best = torch.zeros(W * H, dtype=torch.float64, device=dev)
    who = torch.full((W * H,), 1 << 40, dtype=torch.long, device=dev)
    r = rays.reshape(-1, 3)
    ends = cnt.cumsum(0)
    kept = []
    start = 0
    total = int(ends[-1]) if len(tri) else 0
    while start < len(tri):  # triangles in chunks of at most about 2^24 candidates
        done = int(ends[start - 1]) if start else 0
        stop = int(torch.searchsorted(ends, torch.tensor(done + (1 << 24), device=dev), right=True))
        stop = min(max(stop, start + 1), len(tri)) if done + (1 << 24) < total else len(tri)
        t, n = tri[start:stop], cnt[start:stop]
        k = torch.repeat_interleave(torch.arange(len(t), device=dev), n)
        off = torch.arange(len(k), device=dev) - (n.cumsum(0) - n)[k]
        bw = (i1 - i0 + 1)[t].long()[k]
        pix = (j0[t].long()[k] + off // bw) * W + i0[t].long()[k] + off % bw
        A, ray = a[t], r[pix]
        nrm = torch.linalg.cross(A[:, 1] - A[:, 0], A[:, 2] - A[:, 0])
        d = (nrm * A[:, 0]).sum(1)
        keep = d[k] != 0
        for m in range(3):
            e = torch.linalg.cross(A[:, m], A[:, (m + 1) % 3]) * torch.sign(d)[:, None]
            keep &= (e[k] * ray).sum(1) >= 0
        w = ((nrm / d[:, None])[k] * ray).sum(1)
        keep &= (w > 0) & (w <= 1.0 / cam["near"])
        kept.append((pix[keep], w[keep], t[k[keep]]))
        start = stop
    for pix, w, _ in kept:
        best.scatter_reduce_(0, pix, w, "amax")
    for pix, w, t in kept:
        win = w == best[pix]
        who.scatter_reduce_(0, pix[win], t[win], "amin")
    who = torch.where(best > 0, who, torch.full_like(who, -1))
    return who, 1.0 / best, a


def _cells(dz, mc, sc, valid):
    """Residual, sign and activity of the least-squares surrogate (unit weights)."""
    z, e = torch.zeros_like(dz), torch.full_like(dz, EPS)
    oo, ou, uo = valid & (mc == 0) & (sc == 0), valid & (mc == 0) & (sc == 1), valid & (mc == 1) & (sc == 0)
    r = torch.where(oo, torch.where(dz.abs() <= EPS, dz, e), z)
    r = torch.where(ou, torch.where(dz > 0, z, torch.minimum(-dz, e)), r)
    r = torch.where(uo, torch.where(dz > 0, torch.minimum(dz, e), z), r)
    sgn = torch.where(oo & (dz.abs() <= EPS), torch.ones_like(dz), z)
    sgn = torch.where(ou & (dz <= 0) & (-dz < EPS), -torch.ones_like(dz), sgn)
    return r, torch.where(uo & (dz > 0) & (dz < EPS), torch.ones_like(dz), sgn)


def _sym(J, w):
    H = (J * w[:, None]).T @ J
    return torch.stack([H[u, v] for u in range(6) for v in range(u, 6)])


def _exact_normals(case, s):
    d, c = s["depth"].double(), s["cls"]
    ok = (c == 0) & torch.isfinite(d)
    R = math.ceil(3 * case["sigma"])
    if R:
        x = torch.arange(-R, R + 1, dtype=torch.float64, device=d.device)
        g = torch.exp(-x * x / (2 * case["sigma"] ** 2))
    else:
        g = torch.ones(1, dtype=torch.float64, device=d.device)

    def smooth(q):
        for ax in (1, 2):
            p = torch.nn.functional.pad(q, (R, R, 0, 0) if ax == 2 else (0, 0, R, R))
            q = sum(g[k] * p.narrow(ax, k, q.shape[ax]) for k in range(len(g)))
        return q
    S = smooth(torch.where(ok, d, torch.zeros_like(d))) / smooth(ok.double())
    S = torch.where(ok, S, torch.full_like(S, math.nan))
    zx, zy = torch.full_like(S, math.nan), torch.full_like(S, math.nan)
    zx[:, 1:-1, 1:-1] = 0.5 * (S[:, 1:-1, 2:] - S[:, 1:-1, :-2])
    zy[:, 1:-1, 1:-1] = 0.5 * (S[:, 2:, 1:-1] - S[:, :-2, 1:-1])
    sx, sy = (S / s["cam"]["fx"], S / s["cam"]["fy"]) if case["metric"] else (torch.ones_like(S), torch.ones_like(S))
    nv = torch.stack([sy * zx, zy * sx, -sy * sx], -1)
    nv = nv / nv.norm(dim=-1, keepdim=True)
    return torch.where((torch.isfinite(nv).all(-1) & ok)[..., None], nv, torch.full_like(nv, math.nan))


def exact(case, seed):
    op = case["op"]
    if op in ("icp_align", "dfo_align", "track"):
        return None  # the end of an iteration whose path hangs on each decision
    s = _inputs(case, seed)
    if op == "normals":
        return _exact_normals(case, s)
    cam = s["cam"]
    rays = _rays(cam)
    if cam["model"] == "lidar":
        rays = rays.float().double()  # the table that the framework is given
    if op == "meshify":
        st = case["step"]
        d, c = s["scan"][0].double()[::st, ::st], s["scan"][1][::st, ::st]
        rng_ = torch.where(c == FU, torch.full_like(d, 4.5), d)
        P = torch.as_tensor(s["pose"], device="cuda")
        p = (rng_[..., None] * rays[::st, ::st]) @ P[:3, :3].T + P[:3, 3]
        p = torch.where(((c > 1) | ~torch.isfinite(d))[..., None], P[:3, 3].expand_as(p), p)
        return {"vertices": p.reshape(-1, 3), "faces": None, "labels": None}
    v = torch.as_tensor(s["mesh"][0], device="cuda").double()
    f = torch.as_tensor(s["mesh"][1], device="cuda").long()
    lab = torch.as_tensor(s["mesh"][2], device="cuda").long()
    r = rays.reshape(-1, 3)
    if op != "render":
        sd, sc = s["scan"][0].double().reshape(-1), s["scan"][1].long().reshape(-1)
    out = dict(depth=[], bary=[], e_ls=[], grad=[], jtj=[], cost_l1=[], e2=[], jte=[])
    gv = torch.zeros_like(v)
    graze = 0.0  # the largest share that one pixel has in J^T J
    for pose in s["poses"]:
        who, t, a = _visible(v, f, cam, rays, pose)
        hit = who >= 0
        A = a[who.clamp_min(0)]
        e1, e2 = A[:, 1] - A[:, 0], A[:, 2] - A[:, 0]
        nrm = torch.linalg.cross(e1, e2)
        if op in ("render", "vertex_grad"):
            hp = t[:, None] * r - A[:, 0]
            nn = (nrm * nrm).sum(1)
            b = torch.stack([(torch.linalg.cross(hp, e2) * nrm).sum(1) / nn, (torch.linalg.cross(e1, hp) * nrm).sum(1) / nn], -1)
        if op == "render":
            nan = torch.full_like(t, math.nan)
            out["depth"].append(torch.where(hit, t, nan).reshape(rays.shape[:2]))
            out["bary"].append(torch.where(hit[:, None], b, nan[:, None]).reshape(*rays.shape[:2], 2))
            continue
        nrm = nrm / nrm.norm(dim=1, keepdim=True)
        dz = t - sd
        mc = lab[who.clamp_min(0)]
        valid = hit & (sc < 2) & torch.isfinite(sd)
        if op == "icp_terms":
            m = valid & (sc == 0) & (mc == 0) & (dz.abs() < case["tol"])
            n_, p = nrm[m], sd[m, None] * r[m]
            e = -dz[m] * (n_ * r[m]).sum(1)
            J = torch.cat([n_, torch.linalg.cross(p, n_)], 1)
            out["cost_l1"].append(dz[m].abs().sum())
            out["e2"].append((e * e).sum())
            out["jte"].append((J * e[:, None]).sum(0))
            out["jtj"].append(_sym(J, torch.ones_like(e)))
            continue
        res, sgn = _cells(dz, mc, sc, valid)
        m = sgn != 0
        k = sgn[m] / (nrm[m] * r[m]).sum(1)
        if op == "vertex_grad":
            R = torch.as_tensor(pose[:3, :3], device="cuda")
            nw = nrm[m] @ R.T
            bb = torch.cat([1 - b[m].sum(1, keepdim=True), b[m]], 1)
            for q in range(3):
                gv.index_add_(0, f[who[m], q], (res[m] * k * bb[:, q])[:, None] * nw)
            continue
        J = -torch.cat([nrm[m], t[m, None] * torch.linalg.cross(r[m], nrm[m])], 1) * k[:, None]
        out["e_ls"].append(0.5 * torch.where(valid, res * res, torch.zeros_like(res)).sum())
        out["grad"].append((J * res[m, None]).sum(0))
        out["jtj"].append(_sym(J, torch.ones_like(k)))
        graze = max(graze, float((J * J).sum(1).max()) if len(J) else 0.0)
    if op == "vertex_grad":
        return gv
    ret = {k: torch.stack(q) for k, q in out.items() if q}
    if op.startswith("cost_grad") and graze > 0.02 * float(ret["jtj"].norm()):
        ret["grad"] = ret["jtj"] = None  # they hang on a single pixel at grazing incidence
    ints = {"render": ("tri_id",), "icp_terms": ("n_assoc",)}.get(op, ("counts", "e_table"))
    return {**ret, **{k: None for k in ints}}
