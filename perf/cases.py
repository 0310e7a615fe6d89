"""The work that the framework's speed is judged on: depth maps of one rig
and of many, differentiable depth, fusion of depth maps into voxel maps, and
whole frames from host memory, each through the public entry points.

Inputs are synthetic street canyons (ground, building fronts, parked cars,
value-noise texture, featureless sky) seen by fisheye cameras with
radial-tangential distortion, all made from the seed on the GPU.  ``exact``
restates the paths in 64 bits with plain torch operations.
"""
from __future__ import annotations

import math
from types import SimpleNamespace as NS

import numpy as np
import torch
import torch.nn.functional as TF

import paper_1809_06132_gb300 as P

DEV = "cuda" if torch.cuda.is_available() else "cpu"
T_SOFT = 0.05
MU_VOXELS = 5.0       # truncation in voxels, as in the street and loop workloads
W_MAX = 100.0
LOCAL_HALF = (30.0, 1.5, 30.0)
LOCAL_DROP = 0.6      # the local map's centre below the camera's
CAM_HEIGHT = 1.6
OFFSETS = (-0.5, 0.5, 1.0, -1.0)   # matching cameras along x


# ------------------------------------------------------------------ the cases

def _sweep(name, w, h, cams, **k):
    c = dict(kind="sweep", w=w, h=h, cams=cams, factor=0, window=7, fronto=0, ground=0, crop_w=0, crop_h=0,
             crop_window=9, crop_fronto=0, crop_ground=0, half=False, filters=False, boxes=0)
    c.update(k)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest rig: one matching camera, one level; launches and latency count
        _sweep("sweep-160x128-1cam-32pl", 160, 128, 1, factor=1, window=5, fronto=32),
        # a car's five-camera set-up: half-size level and centre crop, front and
        # ground planes, depth filters and detector boxes
        _sweep("sweep-1024x544-4cam-filtered", 1024, 544, 4, factor=2, window=7, fronto=64, ground=30, crop_w=572,
               crop_h=332, crop_window=9, crop_fronto=64, crop_ground=30, filters=True, boxes=20),
        # the street frame: quarter-size level and full-resolution crop
        _sweep("sweep-1280x1024-2cam", 1280, 1024, 2, factor=4, window=7, fronto=64, ground=32, crop_w=640,
               crop_h=512, crop_window=9, crop_fronto=128, boxes=2),
        # an odd-sized sensor at full resolution, images kept in 16 bits
        _sweep("sweep-1003x751-3cam-half", 1003, 751, 3, factor=1, window=7, fronto=96, half=True, boxes=1),
        # precision mapping: every pixel against 256 planes in three cameras
        _sweep("sweep-1280x1024-3cam-256pl", 1280, 1024, 3, factor=1, window=9, fronto=256, boxes=3),
        # many rigs at once: uneven sweeps of a fleet in one batch
        dict(name="batch-24", kind="batch", n=24, w0=256, w1=640),
        # calibration with gradients: one step on a small rig
        dict(name="soft-96x80-2cam-32pl", kind="soft", w=96, h=80, cams=2, planes=32, window=5),
        # the same at a size that depth learning uses
        dict(name="soft-640x512-2cam-128pl", kind="soft", w=640, h=512, cams=2, planes=128, window=5),
        # a stretch of road fused at 10 cm, its blocks then leaving the local map
        dict(name="fuse-1280x1024-10cm", kind="fuse", w=1280, h=1024, voxel=0.1, frames=8, step=1.0),
        # the same at 2 cm: 25 times the blocks
        dict(name="fuse-1280x1024-2cm", kind="fuse", w=1280, h=1024, voxel=0.02, frames=4, step=0.5),
        # gradients of a fusion step into a dense grid
        dict(name="dense-128x96x136", kind="dense", nx=128, ny=96, nz=136, w=640, h=480, voxel=0.05),
        # live operation: frames from host memory to depth maps in host memory and a map
        dict(name="pipeline-1280x1024", kind="pipe", w=1280, h=1024, cams=2, frames=4, voxel=0.1),
    ]


def _log(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep", "batch", "soft", "fuse", "dense", "pipe"])
    if kind == "sweep":
        w, cams = _log(rng, 160, 1280), rng.randint(1, 4)
        h = max(96, int(w * rng.uniform(0.5, 0.85)))
        extra = dict(half=rng.random() < 0.25, filters=rng.random() < 0.4, boxes=rng.choice([0, 1, 3, 20]))
        if rng.random() < 0.5:   # one full-resolution level, any size
            most = int(256 * 1280 * 1024 * 3 / (w * h * cams))
            return _sweep(None, w, h, cams, factor=1, window=rng.choice([5, 7, 9]),
                          fronto=min(most, _log(rng, 16, 256)), ground=rng.choice([0, 0, 15]), **extra)
        f = rng.choice([2, 4])
        w, h = w // f * f, h // f * f
        return _sweep(None, w, h, cams, factor=f, window=rng.choice([5, 7]), fronto=_log(rng, 16, 96),
                      ground=rng.choice([0, 30, 33]), crop_w=int(w * rng.uniform(0.3, 0.7)),
                      crop_h=int(h * rng.uniform(0.3, 0.7)), crop_window=rng.choice([7, 9]),
                      crop_fronto=_log(rng, 16, 128), crop_ground=rng.choice([0, 30]), **extra)
    if kind == "batch":
        w0 = _log(rng, 160, 400)
        return dict(kind="batch", n=_log(rng, 3, 32), w0=w0, w1=min(640, int(w0 * rng.uniform(1.0, 3.0))))
    if kind == "soft":
        w = _log(rng, 64, 640)
        return dict(kind="soft", w=w, h=max(48, int(w * rng.uniform(0.6, 0.8))), cams=rng.randint(1, 2),
                    planes=_log(rng, 16, 128), window=rng.choice([5, 5, 7]))
    if kind == "fuse":
        w = _log(rng, 320, 1280)
        return dict(kind="fuse", w=w, h=int(w * rng.uniform(0.5, 0.8)), voxel=round(rng.uniform(0.025, 0.2), 3),
                    frames=rng.randint(1, 6), step=round(rng.uniform(0.2, 1.5), 2))
    if kind == "dense":
        w = _log(rng, 160, 640)
        nx, ny, nz = (8 * _log(rng, 4, 16) for _ in range(3))
        return dict(kind="dense", nx=nx, ny=ny, nz=nz, w=w, h=int(w * rng.uniform(0.5, 0.8)),
                    voxel=round(rng.uniform(0.03, 0.12), 3))
    w = _log(rng, 320, 1280) // 4 * 4
    return dict(kind="pipe", w=w, h=int(w * rng.uniform(0.5, 0.8)) // 4 * 4, cams=rng.randint(1, 3),
                frames=rng.randint(2, 5), voxel=round(rng.uniform(0.08, 0.2), 2))


# ------------------------------------------------------------------ rigs and scenes

def _rng(case, seed):
    return np.random.default_rng([seed & 0x7fffffff, case["w"] if "w" in case else case["n"]])


def _camera(g, w, h, f=None):
    while True:
        k1, k2, p1, p2 = (float(v) for v in g.normal(0.0, 0.02, 4))
        s = np.linspace(0.0, 2.5, 51)
        if np.all(1 + 3 * k1 * s + 5 * k2 * s * s - 8 * math.hypot(p1, p2) * np.sqrt(s) > 0.3):
            break
    f = 0.5 * w if f is None else f
    return NS(xi=float(g.uniform(0.8, 1.2)), fx=f, fy=f, cx=w / 2.0, cy=h / 2.0, width=w, height=h, k1=k1, k2=k2,
              p1=p1, p2=p2, r2_max=2.5)


def _rot(pitch, yaw):
    cp, sp, cy, sy = math.cos(pitch), math.sin(pitch), math.cos(yaw), math.sin(yaw)
    return np.array([[cy, 0, sy], [0, 1, 0], [-sy, 0, cy]]) @ np.array([[1, 0, 0], [0, cp, -sp], [0, sp, cp]])


def _rig(g, w, h, cams, f=None):
    ref, cs, poses = _camera(g, w, h, f), [], []
    for j in range(cams):
        cs.append(_camera(g, w, h, f))
        R = _rot(*np.radians(g.uniform(-1.0, 1.0, 2))).T
        poses.append(NS(R=R, t=-R @ np.array([OFFSETS[j], 0.0, 0.0])))
    return NS(ref=ref, cams=cs, ref_to_cam=poses)


def _canyon(g, reach=90.0):
    """Boxes (lo, hi) of a street along z: building fronts and parked cars."""
    out = []
    for side in (-1.0, 1.0):
        z = -12.0
        while z < reach:
            zl, inner, depth, top = g.uniform(8, 20), g.uniform(4.5, 7), g.uniform(3, 8), g.uniform(2, 9)
            x = sorted((side * inner, side * (inner + depth)))
            out.append(((x[0], CAM_HEIGHT - top, z), (x[1], CAM_HEIGHT, z + zl)))
            z += zl + g.uniform(0, 5)
        z = g.uniform(0, 12)
        while z < 0.6 * reach:
            inner, zl = g.uniform(2.4, 3.0), g.uniform(3.8, 4.8)
            x = sorted((side * inner, side * (inner + 1.8)))
            out.append(((x[0], CAM_HEIGHT - 1.5, z), (x[1], CAM_HEIGHT, z + zl)))
            z += zl + g.uniform(6, 20)
    return out


def _rays(cam, x, y, w, h, dtype=torch.float64, ss=1):
    """Unit rays (h ss, w ss, 3) of pixels (x .. x + w, y .. y + h) of cam, and where there is one."""
    o = torch.float64
    u = x + (torch.arange(w * ss, dtype=o, device=DEV) + 0.5) / ss - 0.5
    v = y + (torch.arange(h * ss, dtype=o, device=DEV) + 0.5) / ss - 0.5
    xd, yd = ((u - cam.cx) / cam.fx)[None, :], ((v - cam.cy) / cam.fy)[:, None]
    xd, yd = torch.broadcast_tensors(xd, yd)
    X, Y = xd, yd
    for _ in range(25):
        r2 = X * X + Y * Y
        rad = 1 + cam.k1 * r2 + cam.k2 * r2 * r2
        X, Y = ((xd - 2 * cam.p1 * X * Y - cam.p2 * (r2 + 2 * X * X)) / rad,
                (yd - cam.p1 * (r2 + 2 * Y * Y) - 2 * cam.p2 * X * Y) / rad)
    s = X * X + Y * Y
    disc = 1 + (1 - cam.xi ** 2) * s
    ok = (disc >= 0) & (s <= cam.r2_max)
    f = (cam.xi + disc.clamp_min(0).sqrt()) / (s + 1)
    return torch.stack([f * X, f * Y, f - cam.xi], -1).to(dtype), ok


def _hash(a):
    a = a & 0xffffffff
    a = ((a ^ (a >> 16)) * 0x7FEB352D) & 0xffffffff
    a = ((a ^ (a >> 15)) * 0x446CA68B) & 0xffffffff
    return a ^ (a >> 16)


def _texture(tid, s, t, texel, seed):
    gs, gt = s / texel, t / texel
    i, j = torch.floor(gs), torch.floor(gt)
    fs, ft = gs - i, gt - j
    i, j, base = i.long(), j.long(), _hash(tid * 0x2545F491 + seed)

    def noise(a, b):
        return (_hash(base ^ _hash(a * 0x1B873593 + _hash(b * 0x5BD1E995))) & 0xffff).float() / 65535.0
    lo = (1 - fs) * noise(i, j) + fs * noise(i + 1, j)
    hi = (1 - fs) * noise(i, j + 1) + fs * noise(i + 1, j + 1)
    return 0.1 + 0.8 * ((1 - ft) * lo + ft * hi)


def _cast(boxes, o, d):
    """Ranges (inf = sky) and textured values of the rays o + s d (d unit, flat)."""
    dx, dy, dz = d[:, 0], d[:, 1], d[:, 2]
    best = torch.where(dy > 1e-6, (CAM_HEIGHT - o[1]) / dy.clamp_min(1e-6), torch.full_like(dy, math.inf))
    tid, axis = torch.ones_like(dx, dtype=torch.int64), torch.ones_like(dx, dtype=torch.int64)
    inv = 1.0 / torch.where(d.abs() < 1e-9, torch.full_like(d, 1e-9), d)
    for n, (lo, hi) in enumerate(boxes):
        a = (torch.tensor(lo, device=d.device, dtype=d.dtype) - o) * inv
        b = (torch.tensor(hi, device=d.device, dtype=d.dtype) - o) * inv
        t0, ax = torch.minimum(a, b).max(1)
        hit = (t0 > 1e-3) & (t0 <= torch.maximum(a, b).min(1).values) & (t0 < best)
        best = torch.where(hit, t0, best)
        tid = torch.where(hit, 8 * (n + 2) + ax, tid)
        axis = torch.where(hit, ax, axis)
    return best, tid, axis


def _look(cam, boxes, pose, seed, ss=2):
    """uint8 image of cam at world-to-camera pose, supersampled."""
    r, ok = _rays(cam, 0, 0, cam.width, cam.height, torch.float32, ss)
    R = torch.tensor(np.asarray(pose.R), dtype=torch.float32, device=DEV)
    o = torch.tensor(-np.asarray(pose.R).T @ np.asarray(pose.t), dtype=torch.float32, device=DEV)
    d = r.reshape(-1, 3) @ R
    s, tid, axis = _cast(boxes, o, d)
    hit = torch.isfinite(s)
    p = o + torch.where(hit, s, torch.zeros_like(s))[:, None] * d
    a = torch.where(axis == 0, p[:, 2], p[:, 0])
    b = torch.where(axis == 1, p[:, 2], p[:, 1])
    v = torch.where(hit, _texture(tid, a, b, 0.05, seed), torch.full_like(s, 128 / 255.0))
    v = torch.where(ok.reshape(-1), v, torch.zeros_like(v)).reshape(1, 1, cam.height * ss, cam.width * ss)
    return torch.round(TF.avg_pool2d(v, ss)[0, 0] * 255).clamp(0, 255).to(torch.uint8).contiguous()


def _range(cam, boxes, pose):
    """True range map of cam (0 = none)."""
    r, ok = _rays(cam, 0, 0, cam.width, cam.height, torch.float32)
    R = torch.tensor(np.asarray(pose.R), dtype=torch.float32, device=DEV)
    o = torch.tensor(-np.asarray(pose.R).T @ np.asarray(pose.t), dtype=torch.float32, device=DEV)
    s = _cast(boxes, o, r.reshape(-1, 3) @ R)[0].reshape(cam.height, cam.width)
    return torch.where(ok & torch.isfinite(s), s, torch.zeros_like(s)).contiguous()


def _compose(a, b):
    return NS(R=np.asarray(a.R) @ np.asarray(b.R), t=np.asarray(a.R) @ np.asarray(b.t) + np.asarray(a.t))


def _drive(g, frames, step):
    """World-to-camera poses of a car that drives along z with a little yaw."""
    out = []
    for f in range(frames):
        R = _rot(0.0, math.radians(float(g.uniform(-2, 2))))
        out.append(NS(R=R.T, t=-R.T @ np.array([float(g.uniform(-0.2, 0.2)), 0.0, step * f])))
    return out


def _centre(pose):
    c = -np.asarray(pose.R).T @ np.asarray(pose.t)
    return (float(c[0]), float(c[1]) + LOCAL_DROP, float(c[2]))


def _detections(g, w, h, n):
    out = np.zeros((n, 4), np.int32)
    for i in range(n):
        bw, bh = int(g.uniform(0.02, 0.15) * w), int(g.uniform(0.02, 0.15) * h)
        x, y = int(g.integers(0, w - bw)), int(g.integers(0, h - bh))
        out[i] = (x, y, x + bw, y + bh)
    return out


def _level(kind, window, fronto, ground, near, far, factor=1, crop=(0, 0)):
    sets = [NS(family=0, count=fronto, a=near, b=far, n=(0.0, 0.0, 1.0))] if fronto else []
    if ground:
        sets.append(NS(family=1, count=ground, a=CAM_HEIGHT - 0.5, b=CAM_HEIGHT + 0.5, n=(0.0, 1.0, 0.0)))
    return NS(kind=kind, window=window, factor=factor, crop_w=crop[0], crop_h=crop[1], sets=sets,
              n_planes=sum(s.count for s in sets))


def _levels(c):
    out = []
    if c["factor"]:
        out.append(_level(0, c["window"], c["fronto"], c["ground"], 0.8, 30.0, c["factor"]))
    if c["crop_w"]:
        out.append(_level(1, c["crop_window"], c["crop_fronto"], c["crop_ground"], 1.0, 80.0,
                          crop=(c["crop_w"], c["crop_h"])))
    return out


def _street_levels(w, h):
    """The street frame's two levels at another size."""
    return [_level(0, 7, 64, 32, 0.5, 30.0, 4), _level(1, 9, 128, 0, 1.0, 80.0, crop=(w // 2, h // 2))]


def _filters():
    return NS(enable=True, alpha_upper=0.05, alpha_lower=0.3, split_row=-1.0, ratio_min=1.1, gamma=0.5, delta=0.3,
              window=5)


def _batch_members(c, seed):
    g = _rng(c, seed)
    out = []
    shape = np.random.default_rng(c["n"] * 1009 + c["w0"])   # sizes belong to the case, images to the seed
    for _ in range(c["n"]):
        w = int(round(math.exp(shape.uniform(math.log(c["w0"]), math.log(c["w1"] + 1)))))
        h = int(w * shape.uniform(0.75, 0.8))
        out.append((w, h, int(shape.integers(1, 5)), int(shape.choice([32, 64, 128])), int(shape.integers(0, 4))))
    return g, out


def _voxel_map(c, cam):
    """The map, and the buffers that its blocks are exported to."""
    v = c["voxel"]
    blocks = int(_fuse_blocks(c) * 4) + 4096   # room to spare
    pool = 1 << max(12, math.ceil(math.log2(blocks)))
    export = [torch.zeros((pool // 2, 3), dtype=torch.int32, device=DEV)] + \
             [torch.zeros((pool // 2, 512), dtype=torch.float32, device=DEV) for _ in range(2)]
    return export, P.Tsdf(NS(voxel_size=v, mu=MU_VOXELS * v, w_max=W_MAX, block_dim=8, dense_dim=None, origin=(0.0, 0.0, 0.0),
                     local_half=LOCAL_HALF, hash_slots=4 * pool, pool_blocks=pool), cam)


def _fuse_blocks(c):
    """About the blocks that one frame of such a street updates: the surfaces
    in view inside the local map, cut into block faces (finer blocks miss more
    of the far ones, which few pixels see)."""
    return 1700.0 / (8 * c["voxel"]) ** 1.72


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        g, members = _batch_members(case, seed)
        sweeps, images, boxes = [], [], []
        street = _canyon(g)
        for w, h, cams, planes, nb in members:
            rig = _rig(g, w, h, cams)
            sweeps.append(P.Sweep(rig, [_level(0, 7, planes, 0, 0.5, 30.0)]))
            here = _drive(g, 1, 0.0)[0]
            here.t = here.t - here.R @ np.array([0.0, 0.0, float(g.uniform(0, 20))])
            images.append([_look(rig.ref, street, here, seed, 1)] +
                          [_look(cm, street, _compose(p, here), seed, 1) for cm, p in zip(rig.cams, rig.ref_to_cam)])
            boxes.append(_detections(g, w, h, nb))
        b = P.Batch(sweeps)
        return NS(kind=kind, batch=b, images=images, boxes=boxes, outs=b.alloc_outputs())
    g = _rng(case, seed)
    w, h = case["w"], case["h"]
    street = _canyon(g)
    if kind == "sweep":
        rig = _rig(g, w, h, case["cams"])
        here = _drive(g, 1, 0.0)[0]
        sweep = P.Sweep(rig, _levels(case), filters=_filters() if case["filters"] else None, image_half=case["half"])
        images = [_look(rig.ref, street, here, seed)] + \
                 [_look(cm, street, _compose(p, here), seed) for cm, p in zip(rig.cams, rig.ref_to_cam)]
        return NS(kind=kind, case=case, rig=rig, sweep=sweep, images=images, boxes=_detections(g, w, h, case["boxes"]),
                  out=torch.empty((h, w), dtype=torch.float32, device=DEV), levels=sweep.alloc_level_outputs(DEV))
    if kind == "soft":
        rig = _rig(g, w, h, case["cams"], 0.8 * w)
        here = _drive(g, 1, 0.0)[0]
        images = [_look(c, street, p, seed).float() / 255.0 for c, p in
                  zip([rig.ref] + rig.cams, [here] + [_compose(q, here) for q in rig.ref_to_cam])]
        gr = torch.Generator(device=DEV).manual_seed(seed)
        grads = [torch.randn((h, w), generator=gr, device=DEV) / (w * h) for _ in range(2)]
        soft = P.SoftSweep(rig, _level(0, case["window"], case["planes"], 0, 1.5, 40.0), temperature=T_SOFT)
        return NS(kind=kind, rig=rig, soft=soft, images=[i.requires_grad_() for i in images], grads=grads,
                  delta=torch.zeros((case["cams"], 6), dtype=torch.float64, requires_grad=True))
    if kind == "fuse":
        cam = _camera(g, w, h)
        drive = _drive(g, case["frames"], case["step"])
        export, vmap = _voxel_map(case, cam)
        return NS(kind=kind, poses=drive, depths=[_range(cam, street, p) for p in drive], map=vmap, export=export)
    if kind == "dense":
        v = case["voxel"]
        cam = _camera(g, w, h)
        here = _drive(g, 1, 0.0)[0]
        n = (case["nx"], case["ny"], case["nz"])
        # a grid in front of the camera, standing on the ground
        origin = (-n[0] * v / 2, CAM_HEIGHT + 0.2 - n[1] * v, 1.5)
        grid = NS(dense_dim=n, origin=origin, voxel_size=v, mu=4.0 * v, w_max=W_MAX)
        depth = _range(cam, street, here)
        gr = torch.Generator(device=DEV).manual_seed(seed)
        blocks = n[0] * n[1] * n[2] // 512
        vox = torch.rand((blocks, 512, 2), generator=gr, device=DEV) * 2 - 1
        vox[..., 1] = torch.floor(6 * torch.rand((blocks, 512), generator=gr, device=DEV))   # observations so far
        up = torch.randn((blocks, 512, 2), generator=gr, device=DEV)
        return NS(kind=kind, grid=grid, cam=cam, pose=here, depth=depth.requires_grad_(), vox=vox.requires_grad_(),
                  up=up, delta=torch.zeros(6, dtype=torch.float64, requires_grad=True))
    rig = _rig(g, w, h, case["cams"])
    drive = _drive(g, case["frames"], 1.0)
    frames = [[_look(rig.ref, street, p, seed)] +
              [_look(cm, street, _compose(q, p), seed) for cm, q in zip(rig.cams, rig.ref_to_cam)] for p in drive]
    host = [[i.cpu().pin_memory().numpy() for i in f] for f in frames]
    sweep, (export, vmap) = P.Sweep(rig, _street_levels(w, h)), _voxel_map(case, rig.ref)
    return NS(kind=kind, rig=rig, pipe=P.Pipeline(sweep, vmap), sweep=sweep, map=vmap, export=export, poses=drive,
              frames=host, boxes=[_detections(g, w, h, 2) for _ in drive],
              depths=[np.zeros((h, w), np.float32) for _ in drive])


def _leave(s):
    """Every block leaves the map, as behind a car that is long gone, and goes to the store in the order of the keys."""
    c = _centre(s.poses[-1])
    got = s.map.swap_out((c[0], c[1], c[2] + 1e4))
    k = got[0].long()
    order = torch.argsort((k[:, 2] << 42) + (k[:, 1] << 21) + k[:, 0])
    for a, b in zip(got, s.export):
        torch.index_select(a, 0, order, out=b[:len(a)])
    return s.export


def run(s):
    if s.kind == "sweep":
        s.sweep.depth(s.images, boxes=s.boxes, out=s.out, level_outs=s.levels)
        return [s.out, [[o["depth"], o["c1"], o["c2"], o["kstar"]] for o in s.levels]]
    if s.kind == "batch":
        return s.batch.run(s.images, s.boxes, s.outs)
    if s.kind == "soft":
        rng, cost = P.soft_depth(s.soft, s.images, s.delta)
        return [rng, cost, list(torch.autograd.grad([rng, cost], [s.delta] + s.images, s.grads))]
    if s.kind == "fuse":
        for d, p in zip(s.depths, s.poses):
            s.map.integrate(d, p, _centre(p))
        return _leave(s)
    if s.kind == "dense":
        out = P.dense_fuse(s.vox, s.depth, s.grid, s.cam, s.pose, s.delta)
        return [out, list(torch.autograd.grad(out, [s.vox, s.depth, s.delta], s.up))]
    for f, p, b, d in zip(s.frames, s.poses, s.boxes, s.depths):
        s.pipe.push(f, boxes=b, world_to_ref=p, local_center=_centre(p), depth_out=d)
    s.pipe.flush()
    return [list(s.depths), _leave(s)]


# ------------------------------------------------------------------ what it takes

def _level_px(w, h, lv):
    return (w // lv.factor) * (h // lv.factor) if lv.kind == 0 else lv.crop_w * lv.crop_h


def work(case):
    kind = case["kind"]
    # one plane of one matching camera at one pixel: plane point, rigid
    # transform, projection, distortion, bilinear sample, window statistics,
    # cost and minimum
    unit = 92.0

    def sweep(w, h, cams, levels, outs):
        units = sum(_level_px(w, h, lv) * lv.n_planes * cams for lv in levels)
        px = sum(_level_px(w, h, lv) for lv in levels)
        return (1 + cams) * w * h + 4 * w * h + (16 * px if outs else 0), unit * units
    if kind == "sweep":
        b, f = sweep(case["w"], case["h"], case["cams"], _levels(case), True)
        return dict(bytes=b, flops=f)
    if kind == "batch":
        got = [sweep(w, h, cams, [_level(0, 7, planes, 0, 0.5, 30.0)], False)
               for w, h, cams, planes, _ in _batch_members(case, 0)[1]]
        return dict(bytes=sum(b for b, _ in got), flops=sum(f for _, f in got))
    if kind == "soft":
        px, n = case["w"] * case["h"], 1 + case["cams"]
        # forward as above; backward: the sample again with its pose derivative,
        # the coefficients' box sums, the chain to the four texels and the pose
        units = px * case["planes"] * case["cams"]
        return dict(bytes=px * (4 * n + 8 + 8 + 4 * n), flops=units * (unit + 170.0))
    if kind == "dense":
        vox, px = case["nx"] * case["ny"] * case["nz"], case["w"] * case["h"]
        return dict(bytes=vox * (8 + 8 + 8 + 8) + px * 8, flops=vox * 140.0)
    px = case["w"] * case["h"]
    step = case.get("step", 1.0)
    # per frame the depth map and the blocks in view, read and written; at the end every block once
    touched = _fuse_blocks(case)
    held = touched * (1 + step * (case["frames"] - 1) / 30.0)
    b = case["frames"] * (4 * px + touched * 512 * 16) + held * 512 * 16
    f = case["frames"] * touched * 512 * 60.0
    if kind == "pipe":
        sb, sf = sweep(case["w"], case["h"], case["cams"], _street_levels(case["w"], case["h"]), False)
        b, f = b + case["frames"] * sb, f + case["frames"] * sf
    return dict(bytes=b, flops=f)


# ------------------------------------------------------------------ in 64 bits

D64 = torch.float64


def _t(a):
    return torch.tensor(np.asarray(a, dtype=np.float64), device=DEV)


def _scaled(c, s):
    return NS(**{**vars(c), "fx": c.fx / s, "fy": c.fy / s, "cx": (c.cx - (s - 1) / 2.0) / s,
                 "cy": (c.cy - (s - 1) / 2.0) / s, "width": c.width // s, "height": c.height // s})


def _project(cam, X):
    n = X.square().sum(-1).sqrt()
    den = X[..., 2] + cam.xi * n
    x, y = X[..., 0] / den, X[..., 1] / den
    r2 = x * x + y * y
    rad = 1 + cam.k1 * r2 + cam.k2 * r2 * r2
    u = cam.fx * (x * rad + 2 * cam.p1 * x * y + cam.p2 * (r2 + 2 * x * x)) + cam.cx
    v = cam.fy * (y * rad + cam.p1 * (r2 + 2 * y * y) + 2 * cam.p2 * x * y) + cam.cy
    lim = min(cam.xi, 1 / cam.xi) if cam.xi > 0 else 0.0
    return u, v, (X[..., 2] > -lim * n) & (r2 <= cam.r2_max)


def _bilinear(img, u, v, ok):
    H, W = img.shape
    ok = ok & (u >= 0) & (u <= W - 1) & (v >= 0) & (v <= H - 1)
    u, v = torch.where(ok, u, torch.zeros_like(u)), torch.where(ok, v, torch.zeros_like(v))
    x0, y0 = u.detach().floor().long(), v.detach().floor().long()
    x1, y1 = (x0 + 1).clamp_max(W - 1), (y0 + 1).clamp_max(H - 1)
    a, b = u - x0, v - y0
    flat = img.reshape(-1)
    top = (1 - a) * flat[y0 * W + x0] + a * flat[y0 * W + x1]
    bot = (1 - a) * flat[y1 * W + x0] + a * flat[y1 * W + x1]
    return (1 - b) * top + b * bot, ok


def _box(x, win):
    return TF.avg_pool2d(x[None, None], win, 1)[0, 0] * (win * win)


def _cost(ref, w, ok, win):
    """(1 - ZNCC) / 2 of every window inside the image (inf = invalid), padded to the image."""
    n, p = win * win, win // 2
    bad = _box((~ok).to(D64), win) > 0.5
    w = torch.where(ok, w, torch.zeros_like(w))
    sr, sw = _box(ref, win), _box(w, win)
    vr = _box(ref * ref, win) - sr * sr / n
    vw = _box(w * w, win) - sw * sw / n
    good = ~bad & (vr.detach() >= n * 1e-8) & (vw.detach() >= n * 1e-8)
    one = torch.ones_like(vr)
    z = (_box(ref * w, win) - sr * sw / n) / (torch.where(good, vr, one) * torch.where(good, vw, one)).sqrt()
    c = torch.where(good, (0.5 * (1 - z)).clamp(0, 1), torch.full_like(z, math.inf))
    return TF.pad(c, (p, p, p, p), value=math.inf)


def _planes(lv):
    out = []
    for si, s in enumerate(lv.sets):
        for i in range(s.count):
            t = i / (s.count - 1) if s.count > 1 else 0.0
            out.append((si, i, (s.n if s.family else (0.0, 0.0, 1.0)),
                        s.a + t * (s.b - s.a) if s.family else 1 / (1 / s.b + t * (1 / s.a - 1 / s.b))))
    return out


def _warp(rays, has, n, d, R, t, cam, img):
    nr = rays @ _t(n)
    X = (d / torch.where(nr > 0, nr, torch.ones_like(nr)))[..., None] * (rays @ R.T) + t
    u, v, ok = _project(cam, X)
    return _bilinear(img, u, v, ok & has & (nr > 0))


def _exact_level(rig, lv, images, half):
    """Depth, best and second-best cost of one level."""
    ref8 = images[0].to(D64)
    if lv.kind == 0:
        f = lv.factor
        shrink = lambda i: TF.avg_pool2d(i.to(D64)[None, None], f)[0, 0] / 255.0 - 0.5  # noqa: E731
        rc, cams = _scaled(rig.ref, f), [_scaled(c, f) for c in rig.cams]
        ref, imgs, x0, y0 = shrink(ref8), [shrink(i) for i in images[1:]], 0, 0
        rw, rh = rc.width, rc.height
    else:
        x0, y0 = (rig.ref.width - lv.crop_w) // 2, (rig.ref.height - lv.crop_h) // 2
        rc, cams, rw, rh = rig.ref, rig.cams, lv.crop_w, lv.crop_h
        ref = ref8[y0:y0 + rh, x0:x0 + rw] / 255.0 - 0.5
        imgs = [i.to(D64) / 255.0 - 0.5 for i in images[1:]]
    if half:
        imgs = [i.half().to(D64) for i in imgs]
    rays, has = _rays(rc, x0, y0, rw, rh)
    planes = _planes(lv)
    vol = torch.full((len(planes), rh, rw), math.inf, dtype=D64, device=DEV)
    for k, (_, _, n, d) in enumerate(planes):
        for cam, pose, img in zip(cams, rig.ref_to_cam, imgs):
            w, ok = _warp(rays, has, n, d, _t(pose.R), _t(pose.t), cam, img)
            vol[k] = torch.minimum(vol[k], _cost(ref, w, ok, lv.window))
    c1, kb = vol.min(0)
    won = torch.isfinite(c1)
    second = vol.scatter(0, kb[None], math.inf).min(0).values
    idx = torch.tensor([i for _, i, _, _ in planes], device=DEV)[kb]
    sid = torch.tensor([s for s, _, _, _ in planes], device=DEV)[kb]
    count = torch.tensor([s.count for s in lv.sets], device=DEV)[sid]
    cm = vol.gather(0, (kb - 1).clamp_min(0)[None])[0]
    cp = vol.gather(0, (kb + 1).clamp_max(len(planes) - 1)[None])[0]
    den = cm - 2 * c1 + cp
    fit = (idx > 0) & (idx < count - 1) & torch.isfinite(cm) & torch.isfinite(cp) & (den > 0)
    delta = torch.where(fit, ((cm - cp) / (2 * den)).clamp(-0.5, 0.5), torch.zeros_like(c1))
    t = torch.where(count > 1, (idx + delta) / (count - 1).clamp_min(1), torch.zeros_like(c1))
    depth = torch.zeros_like(c1)
    for si, s in enumerate(lv.sets):
        n = _t(s.n if s.family else (0.0, 0.0, 1.0))
        p = s.a + t * (s.b - s.a) if s.family else 1 / (1 / s.b + t * (1 / s.a - 1 / s.b))
        depth = torch.where(won & (sid == si), p / (rays @ n), depth)
    return depth, c1, second


def _exact_depth(rig, levels, images, boxes, filters=False, half=False):
    H, W = images[0].shape
    out, got = torch.zeros((H, W), dtype=D64, device=DEV), []
    row = torch.arange(H, device=DEV, dtype=D64)[:, None]

    def keep(c1, c2, r):
        alpha = torch.where(r < H / 2, 0.05, 0.3)
        return (c1 <= alpha) & (c2 >= 1.1 * c1)
    for lv in levels:
        depth, c1, c2 = _exact_level(rig, lv, images, half)
        got.append([depth, c1, c2, None])
        d = depth
        if lv.kind == 0:
            f = lv.factor
            if filters:
                d = torch.where(keep(c1, c2, f * row[:depth.shape[0]] + 0.5 * (f - 1)), d, torch.zeros_like(d))
            out = d.repeat_interleave(f, 0).repeat_interleave(f, 1)
        else:
            x0, y0 = (W - lv.crop_w) // 2, (H - lv.crop_h) // 2
            ok = d > 0
            if filters:
                ok &= keep(c1, c2, row[y0:y0 + lv.crop_h])
            view = out[y0:y0 + lv.crop_h, x0:x0 + lv.crop_w]
            view.copy_(torch.where(ok, d, view))
    if filters:
        same, seen = torch.zeros_like(out), torch.zeros_like(out)
        pad, inside = TF.pad(out, (2, 2, 2, 2)), TF.pad(torch.ones_like(out), (2, 2, 2, 2))
        for dy in range(5):
            for dx in range(5):
                if dx == 2 and dy == 2:
                    continue
                o = pad[dy:dy + H, dx:dx + W]
                seen += inside[dy:dy + H, dx:dx + W]
                same += ((o > 0) & ((o - out).abs() < 0.5)).to(D64)
        out = torch.where(same >= 0.3 * seen, out, torch.zeros_like(out))
    for x0, y0, x1, y1 in np.asarray(boxes).tolist():
        out[y0:y1, x0:x1] = 0
    return out, got


def _exact_soft(s, case):
    rig, win = s.rig, case["window"]
    lv = _level(0, win, case["planes"], 0, 1.5, 40.0)
    rays, has = _rays(rig.ref, 0, 0, rig.ref.width, rig.ref.height)
    imgs = [i.detach().to(D64).requires_grad_() for i in s.images]
    delta = torch.zeros((len(rig.cams), 6), dtype=D64, device=DEV, requires_grad=True)

    def pose(j):   # first order in delta, which is all its gradient at zero takes
        R, t = _t(rig.ref_to_cam[j].R), _t(rig.ref_to_cam[j].t)
        x, y, z = delta[j, 0], delta[j, 1], delta[j, 2]
        o = torch.zeros_like(x)
        K = torch.stack([o, -z, y, z, o, -x, -y, x, o]).reshape(3, 3)
        return R + K @ R, t + K @ t + delta[j, 3:]

    def costs(n, d):
        each = []
        for j, cam in enumerate(rig.cams):
            R, t = pose(j)
            w, ok = _warp(rays, has, n, d, R, t, cam, imgs[1 + j])
            each.append(_cost(imgs[0], w, ok, win))
        return torch.stack(each).min(0).values

    planes = _planes(lv)
    with torch.no_grad():
        vol = torch.stack([costs(n, d) for _, _, n, d in planes])
    some = torch.isfinite(vol).any(0) & has
    C = torch.where(torch.isfinite(vol), vol, torch.full_like(vol, 1e3)).requires_grad_()
    rho = torch.stack([(rays @ _t(n)) / d for _, _, n, d in planes])
    share = torch.softmax(-C / T_SOFT, 0)
    zero = torch.zeros((), dtype=D64, device=DEV)
    rng = torch.where(some, 1 / (share * rho).sum(0), zero)
    cost = torch.where(some, -T_SOFT * torch.logsumexp(-C / T_SOFT, 0), zero)
    gC, = torch.autograd.grad([rng, cost], C, [g.to(D64) for g in s.grads])
    gC = torch.where(torch.isfinite(vol) & some, gC, zero)
    wrt = [delta] + imgs
    total = [torch.zeros_like(x) for x in wrt]
    for k, (_, _, n, d) in enumerate(planes):
        c = costs(n, d)
        c = torch.where(torch.isfinite(c), c, zero)
        for a, b in zip(total, torch.autograd.grad((c * gC[k]).sum(), wrt)):
            a += b
    return [rng.detach(), cost.detach(), [total[0].cpu()] + total[1:]]


def _exact_dense(s, case):
    v, mu = case["voxel"], 4.0 * case["voxel"]
    n = (case["nx"], case["ny"], case["nz"])
    b = torch.arange(n[0] * n[1] * n[2] // 512, device=DEV)[:, None]
    q = torch.arange(512, device=DEV)[None, :]
    nb = (n[0] // 8, n[1] // 8)
    at = torch.stack([b % nb[0] * 8 + q % 8, b // nb[0] % nb[1] * 8 + q // 8 % 8, b // (nb[0] * nb[1]) * 8 + q // 64], -1)
    Xw = _t(s.grid.origin) + (at.to(D64) + 0.5) * v
    R, t = _t(s.pose.R), _t(s.pose.t)
    X = Xw @ R.T + t
    u, w, ok = _project(s.cam, X)
    u, w = torch.floor(u + 0.5), torch.floor(w + 0.5)
    ok &= (u >= 0) & (w >= 0) & (u < s.cam.width) & (w < s.cam.height)
    pix = torch.where(ok, w * s.cam.width + u, torch.zeros_like(u)).long()
    d = s.depth.detach().to(D64).reshape(-1)[pix]
    far = X.square().sum(-1).sqrt()
    eta = d - far
    ok &= (d > 0) & (eta >= -mu)
    old, obs = s.vox.detach()[..., 0].to(D64), s.vox.detach()[..., 1].to(D64)
    D = torch.where(ok, (obs * old + (eta / mu).clamp_max(1.0)) / (obs + 1), old)
    Wn = torch.where(ok, (obs + 1).clamp_max(W_MAX), obs)
    g = s.up[..., 0].to(D64)
    gv = torch.stack([torch.where(ok, g * obs / (obs + 1), g), torch.zeros_like(g)], -1)
    ge = torch.where(ok & (eta < mu), g / (mu * (obs + 1)), torch.zeros_like(g))
    gd = torch.zeros(s.depth.numel(), dtype=D64, device=DEV).index_add_(0, pix.reshape(-1), ge.reshape(-1))
    gx = -(ge / far)[..., None] * X
    gp = torch.cat([torch.cross(X, gx, dim=-1).sum((0, 1)), gx.sum((0, 1))])
    return [torch.stack([D, Wn], -1), [gv, gd.reshape(s.depth.shape), gp.cpu()]]


def exact(case, seed):
    kind = case["kind"]
    # fusion into hashed blocks returns the blocks that a decision in 32 bits
    # picked: there is no other list of the same blocks to compare it with
    if kind == "fuse":
        return None
    s = prepare(case, seed)
    if kind == "sweep":
        d, got = _exact_depth(s.rig, _levels(case), s.images, s.boxes, case["filters"], case["half"])
        return [d, got]
    if kind == "batch":
        return [_exact_depth(sw.rig, sw.levels, im, b)[0] for sw, im, b in zip(s.batch.sweeps, s.images, s.boxes)]
    if kind == "soft":
        return _exact_soft(s, case)
    if kind == "dense":
        return _exact_dense(s, case)
    up = [[torch.from_numpy(i).to(DEV) for i in f] for f in s.frames]
    levels = _street_levels(case["w"], case["h"])
    return [[_exact_depth(s.rig, levels, f, b)[0] for f, b in zip(up, s.boxes)], [None, None, None]]
