"""Measured workloads of the tracking library: what its users run, over the sizes they run it at.

A case is a dict of plain values. Four kinds, each through the public entry
points of the package:

* ``track``     a depth frame (or a batch of independent ones) is set and aligned
                to its model: kf_set_frame(_batch), then kf_align(_batch);
* ``localise``  one frame of tracking against a finished map: set the frame,
                align it, raycast the map at the estimated pose, and make that
                raycast the next model;
* ``map``       the mapping half of a frame: integrate a depth frame into the
                volume and raycast the volume at the same pose;
* ``reduce``    the allocation-free normal-equation sums on the caller's maps.

Inputs are drawn on the GPU from the seed alone: a furnished room seen by a
Kinect-like camera, with its depth noise, dropout and uniform outliers.
``exact`` restates each kind in 64 bits with plain torch; the discrete choices
(matched pixel, histogram bin, voxel pixel, sign changes) are the float32
decisions the library documents, everything summed or solved is float64.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1802_03980_gb300 as kf

F32, F64 = torch.float32, torch.float64
NAN = float("nan")

# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
# sizes of a mixed batch, largest share first to last in equal parts
MIXED_SIZES = ((320, 240), (640, 480), (960, 720), (1280, 960))
MOST_BATCH_PIXELS = 256 * 640 * 480


def _track(name=None, pairs=1, width=640, height=480, mixed=False, levels=3, fp16=False,
           source="device", mode="paper", outliers=0.10, lam=1e3):
    c = dict(kind="track", pairs=pairs, width=width, height=height, mixed=mixed, levels=levels,
             fp16=fp16, source=source, mode=mode, outliers=outliers, lam=lam)
    return dict(c, name=name) if name else c


def _map(name=None, kind="map", width=640, height=480, res=512, frames=3):
    c = dict(kind=kind, width=width, height=height, res=res, frames=frames)
    return dict(c, name=name) if name else c


def _reduce(name=None, width=640, height=480, khi=255, noise=1.0):
    c = dict(kind="reduce", width=width, height=height, khi=khi, noise=noise)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a low-resolution sensor, one pyramid level; latency only
        _track("track_160x120_l1", width=160, height=120, levels=1, outliers=0.0),
        # the ordinary call: one Kinect frame, tracked as it arrives, already on the GPU
        _track("track_640x480"),
        # the same from page-locked host memory into half-precision maps
        _track("track_640x480_host_fp16", fp16=True, source="pinned"),
        # odd size, and the original KinectFusion loop as the paper compares with it: no
        # seed, no filter, fixed iteration counts, normal-angle gate
        _track("track_333x251_original", width=333, height=251, mode="original", lam=0.0,
               outliers=0.02),
        # one frame of the largest sensor
        _track("track_1280x960", width=1280, height=960),
        # a serving step: a batch of frames that arrives in page-locked host memory
        _track("batch32_640x480_host", pairs=32, source="pinned"),
        # independent cameras of different resolutions in one batch, half-precision maps
        _track("batch64_mixed_fp16", pairs=64, mixed=True, fp16=True, outliers=0.15),
        # the throughput workload: many independent frame-to-model pairs
        _track("batch256_640x480", pairs=256),
        # the paper's own normals and association: integral images and normal shooting
        _track("batch16_shooting", pairs=16, mode="shooting", outliers=0.0),
        # sums for a caller that may not allocate
        _reduce("reduce_640x480"),
        # the mapping half of a frame, the paper's 512^3 cube
        _map("map_512_640x480"),
        # tracking inside a finished map, model raycast at every frame
        _map("localise_512_640x480", kind="localise", frames=6),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo=120, hi=1280):
    """A frame size: width over the whole range, often odd; height 3/4 of it or near."""
    w = _log(rng, lo, hi)
    h = max(90, int(w * rng.choice((0.75, 0.75, 0.5625, rng.uniform(0.5, 0.9)))))
    return w, h


def draw(rng):
    kind = rng.choice(("one", "one", "batch", "batch", "batch", "reduce", "map", "localise"))
    w, h = _size(rng)
    if kind == "reduce":
        return _reduce(width=w, height=h, khi=_log(rng, 20, 511), noise=rng.choice((0.5, 1.0, 2.0)))
    if kind in ("map", "localise"):
        return _map(kind=kind, width=w, height=h, res=_log(rng, 128, 512), frames=rng.randint(2, 6))
    mode = rng.choice(("paper", "paper", "paper", "original", "shooting"))
    outl = 0.0 if mode == "shooting" else rng.choice((0.0, 0.05, 0.10, 0.15))
    pairs, mixed = 1, False
    if kind == "batch":
        mixed = mode == "paper" and rng.random() < 0.3
        most = 64 if mixed else max(2, min(256, MOST_BATCH_PIXELS // (w * h)))
        if mode == "shooting":
            most = max(2, min(most, 16 * 640 * 480 // (w * h)))
        elif mode == "original":
            most = max(2, most // 3)
        pairs = _log(rng, 2, most)
    return _track(pairs=pairs, width=w, height=h, mixed=mixed, levels=rng.choice((1, 2, 3, 3, 3, 4)),
                  fp16=rng.random() < 0.4, source=rng.choice(("device", "device", "pinned")),
                  mode=mode, outliers=outl,
                  lam=0.0 if mode == "original" else float(10 ** rng.uniform(0.7, 3.0)))


# ---------------------------------------------------------------------------
# inputs: a furnished room, ray-cast on the GPU
# ---------------------------------------------------------------------------
def _rotation(axis, deg):
    a = np.asarray(axis, np.float64)
    a = a / np.linalg.norm(a)
    K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    t = math.radians(deg)
    return np.eye(3) + math.sin(t) * K + (1 - math.cos(t)) * (K @ K)


def _pose(R, t):
    T = np.eye(4)
    T[:3, :3] = R
    T[:3, 3] = t
    return T


def _look_at(eye, target):
    eye = np.asarray(eye, np.float64)
    z = np.asarray(target, np.float64) - eye
    z /= np.linalg.norm(z)
    x = np.cross([0.0, 1.0, 0.0], z)
    x /= np.linalg.norm(x)
    return _pose(np.stack([x, np.cross(z, x), z], axis=1), eye)


def _camera(w, h):
    f = 525.0 * w / 640.0  # the Kinect's field of view
    return (w, h, f, f, (w - 1) / 2.0, (h - 1) / 2.0)


def _room(rng):
    """Walls as axis-aligned planes (axis, offset, side), spheres and boxes within 4 m."""
    u = rng.uniform
    walls = [(1, u(1.0, 1.4)), (1, -u(1.3, 1.7)), (2, u(3.2, 3.8)), (0, -u(1.8, 2.4)), (0, u(1.8, 2.4))]
    balls = [((u(-1.0, -0.4), u(-0.4, 0.5), u(1.6, 2.6)), u(0.2, 0.4)),
             ((u(0.4, 1.0), u(-0.4, 0.5), u(1.4, 2.4)), u(0.15, 0.35))]
    lo = (u(-0.3, 0.3), u(0.2, 0.6), u(2.0, 2.8))
    boxes = [(lo, tuple(c + u(0.3, 0.6) for c in lo))]
    return walls, balls, boxes


def _cast(room, T, K):
    """Camera-frame depth, world points and world normals of every pixel (float64)."""
    w, h, fx, fy, cx, cy = K
    dev = "cuda"
    u = (torch.arange(w, device=dev, dtype=F64) - cx) / fx
    v = (torch.arange(h, device=dev, dtype=F64) - cy) / fy
    R, o = T[:3, :3], T[:3, 3]
    d = [R[a, 0] * u[None, :] + (R[a, 1] * v[:, None] + R[a, 2]) for a in range(3)]
    best = torch.full((h, w), math.inf, device=dev, dtype=F64)
    n = [torch.full((h, w), NAN, device=dev, dtype=F64) for _ in range(3)]

    def take(s, ok, normal):
        nonlocal best, n
        ok = ok & (s > 1e-9) & (s < best)
        best = torch.where(ok, s, best)
        n = [torch.where(ok, normal[a], n[a]) for a in range(3)]

    walls, balls, boxes = room
    zero = torch.zeros((), device=dev, dtype=F64)
    for axis, off in walls:
        s = (off - o[axis]) / d[axis]
        side = [zero] * 3
        side[axis] = -torch.sign(d[axis])
        take(s, torch.isfinite(s), side)
    dd = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
    for c, r in balls:
        oc = [o[a] - c[a] for a in range(3)]
        b = d[0] * oc[0] + d[1] * oc[1] + d[2] * oc[2]
        disc = b * b - dd * (sum(x * x for x in oc) - r * r)
        s = (-b - torch.sqrt(disc.clamp(min=0))) / dd
        take(s, disc >= 0, [(oc[a] + s * d[a]) / r for a in range(3)])
    for lo, hi in boxes:
        t1, t2 = [(lo[a] - o[a]) / d[a] for a in range(3)], [(hi[a] - o[a]) / d[a] for a in range(3)]
        near = torch.stack([torch.minimum(a, b) for a, b in zip(t1, t2)])
        far = torch.stack([torch.maximum(a, b) for a, b in zip(t1, t2)])
        tin, axis = near.max(0)
        take(tin, tin <= far.min(0).values, [torch.where(axis == a, -torch.sign(d[a]), zero) for a in range(3)])
    p = torch.stack([o[a] + best * d[a] for a in range(3)], -1)
    return best, p, torch.stack(n, -1)


def _sense(depth, gen, outliers=0.0, dropout=0.02, noise=1.0):
    """What the sensor reports of a true depth: float32 metres, 0 where it has none."""
    z = torch.where(torch.isfinite(depth), depth, torch.zeros_like(depth))
    r = torch.rand((3,) + z.shape, generator=gen, device=z.device, dtype=F32).to(F64)
    g = torch.randn(z.shape, generator=gen, device=z.device, dtype=F32).to(F64)
    z = z + noise * g * (0.0012 + 0.0019 * (z - 0.4) ** 2)
    z = torch.where(r[0] < outliers, 0.5 + 3.5 * r[1], z)
    z = torch.where((r[2] < dropout) | (z < 0.25), torch.zeros_like(z), z)
    return z.to(F32).contiguous()


def _motion(rng, deg, metres):
    def unit():
        v = np.array([rng.gauss(0, 1) for _ in range(3)])
        return v / np.linalg.norm(v)
    return _pose(_rotation(unit(), rng.uniform(0, deg)), rng.uniform(0, metres) * unit()), _rotation(unit(), 0.3)


def _caps(c):
    return (10, 5, 4, 4)[: c["levels"]]


def _params(c):
    p = kf.kf_default_params()
    p.levels = c["levels"]
    for i, m in enumerate(_caps(c)):
        p.max_iters[i] = m
    p.precision = kf.KF_FP16 if c["fp16"] else kf.KF_FP32
    if c["mode"] == "original":
        p.flags = 0
        p.cos_angle_min = math.cos(math.radians(20.0))
    elif c["mode"] == "shooting":
        p.normal_mode = kf.KF_NORMALS_INTEGRAL
        p.shoot_radius = 2
    return p


def _sizes(c):
    if not c["mixed"]:
        return [(c["width"], c["height"])] * c["pairs"]
    n = c["pairs"]
    return [MIXED_SIZES[i * len(MIXED_SIZES) // n] for i in range(n)]


def _pairs(c, seed):
    """The case's frames, models, poses and priors."""
    rng = random.Random(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    # a loop without a seed has to start near: it tracks a camera at frame rate
    deg, metres = (1.5, 0.015) if c["mode"] == "original" else (5.0, 0.05)
    rooms = [_room(rng) for _ in range(4)]
    out = []
    for i, (w, h) in enumerate(_sizes(c)):
        room = rooms[i % 4]
        K = _camera(w, h)
        base = _look_at([rng.uniform(-0.1, 0.1) for _ in range(3)],
                        (rng.uniform(-0.2, 0.2), rng.uniform(-0.1, 0.1), 3.0))
        dT, prior_noise = _motion(rng, deg, metres)
        truth = base @ dT
        depth = _sense(_cast(room, truth, K)[0], gen, c["outliers"])
        _, mv, mn = _cast(room, base, K)
        out.append(dict(K=K, depth=depth, mv=mv.to(F32).contiguous(), mn=mn.to(F32).contiguous(),
                        base=base, prior=prior_noise @ truth[:3, :3]))
    return out


class _State:
    """What the caller holds between calls; releases its handles when dropped."""

    def __init__(self):
        self.trackers, self.volume = [], None

    def __del__(self):
        for t in self.trackers:
            kf.kf_track_destroy(t)
        if self.volume is not None:
            kf.kf_volume_destroy(self.volume)


def _prepare_track(c, seed):
    pairs = _pairs(c, seed)
    p = _params(c)
    s = _State()
    s.kind, s.n, s.lam = "track", len(pairs), [c["lam"]] * len(pairs)
    s.Ks = [pr["K"] for pr in pairs]
    s.frames = [pr["depth"].cpu().pin_memory() if c["source"] == "pinned" else pr["depth"] for pr in pairs]
    s.ptrs = [f.data_ptr() for f in s.frames]
    s.source = kf.KF_FRAME_HOST if c["source"] == "pinned" else kf.KF_FRAME_DEVICE
    s.priors = np.stack([pr["prior"] for pr in pairs])
    s.inits = np.stack([pr["base"] for pr in pairs])
    s.stream = torch.cuda.Stream()
    torch.cuda.synchronize()  # the inputs are made on another stream
    for pr in pairs:
        w, h = pr["K"][:2]
        t = kf.kf_track_create(p, w, h, s.stream.cuda_stream)
        s.trackers.append(t)
        kf.kf_set_model(t, pr["mv"].data_ptr(), pr["mn"].data_ptr(), pr["base"], pr["K"], True)
    torch.cuda.synchronize()  # the models are copied: their inputs may go
    return s


def _walk(c, seed):
    """A camera's path through a room, the frames it sees, and the volume they go into."""
    rng = random.Random(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    room = _room(rng)
    K = _camera(c["width"], c["height"])
    vp = kf.kf_volume_default_params()
    vp.res = c["res"]
    vp.side = 6.0
    vp.origin[0], vp.origin[1], vp.origin[2] = -3.0, -3.0, -1.0
    vp.mu = max(0.05, 4.0 * 6.0 / c["res"])
    path = [_look_at((0.05 * math.sin(k + 1.0), 0.03 * k - 0.05, 0.02 * k),
                     (rng.uniform(-0.15, 0.15), rng.uniform(-0.1, 0.1), 3.0))
            for k in range(c["frames"] + 1)]
    return vp, K, path, [_sense(_cast(room, T, K)[0], gen, dropout=0.01, noise=0.5) for T in path]


RAY = (0.4, 5.0)


def _step(vp):
    return min(0.02, 0.5 * vp.mu)


def _prepare_map(c, seed):
    s = _State()
    s.kind, s.stream = c["kind"], torch.cuda.Stream()
    vp, s.K, path, depths = _walk(c, seed)
    torch.cuda.synchronize()  # the frames are made on another stream
    s.volume = kf.kf_volume_create(vp, s.stream.cuda_stream)
    for D, T in zip(depths[:-1], path[:-1]):
        kf.kf_volume_integrate(s.volume, D.data_ptr(), s.K, T, True)
    s.dz = _step(vp)
    s.depth, s.pose = depths[-1], path[-1]
    shape = (c["height"], c["width"], 3)
    s.V = torch.empty(shape, device="cuda", dtype=F32)
    s.N = torch.empty(shape, device="cuda", dtype=F32)
    if c["kind"] == "localise":
        s.prior, s.init, s.lam = path[-1][:3, :3], path[-2], 5.0
        t = kf.kf_track_create(kf.kf_default_params(), c["width"], c["height"], s.stream.cuda_stream)
        s.trackers.append(t)
        kf.kf_volume_raycast(s.volume, s.K, s.init, RAY[0], RAY[1], s.dz, s.V.data_ptr(), s.N.data_ptr(), True)
        kf.kf_set_model(t, s.V.data_ptr(), s.N.data_ptr(), s.init, s.K, True)
    torch.cuda.synchronize()
    return s


def _prepare_reduce(c, seed):
    pr = _pairs(dict(kind="track", pairs=1, width=c["width"], height=c["height"], mixed=False, mode="paper",
                     outliers=0.05), seed)[0]
    s = _State()
    s.kind, s.K, s.khi = "reduce", pr["K"], c["khi"]
    w, h, fx, fy, cx, cy = pr["K"]
    z = pr["depth"]
    u = torch.arange(w, device="cuda", dtype=F32) - cx
    v = torch.arange(h, device="cuda", dtype=F32) - cy
    fv = torch.stack([u[None, :] * z / fx, v[:, None] * z / fy, z], -1)
    s.fv = torch.where((z > 0)[..., None], fv, torch.full_like(fv, NAN)).contiguous()
    s.mv, s.mn, s.model_pose = pr["mv"], pr["mn"], pr["base"]
    s.pose = pr["base"].copy()
    s.pose[:3, :3] = pr["prior"]
    s.sums = torch.zeros(29, device="cuda", dtype=F64)
    s.stream = torch.cuda.current_stream().cuda_stream
    return s


def prepare(case, seed):
    make = {"track": _prepare_track, "map": _prepare_map, "localise": _prepare_map, "reduce": _prepare_reduce}
    return make[case["kind"]](case, seed)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def _results(res):
    """kf_result records as (whole-number fields, rms residual) arrays."""
    raw = np.frombuffer(b"".join(bytes(r) for r in res), np.uint8).reshape(len(res), -1)
    counts = raw[:, :48].copy().view(np.int32)
    return counts, raw[:, 48:56].copy().view(np.float64)[:, 0]


def run(s):
    if s.kind == "track":
        if s.n == 1:
            t = s.trackers[0]
            kf.kf_set_frame(t, s.ptrs[0], s.Ks[0], s.source)
            status, pose, res = kf.kf_align(t, s.priors[0], s.inits[0], s.lam[0])
            res = [res]
        else:
            kf.kf_set_frame_batch(s.trackers, s.ptrs, s.Ks, s.source)
            status, pose, res = kf.kf_align_batch(s.trackers, s.priors, s.inits, s.lam)
        counts, rms = _results(res)
        return {"status": status, "pose": pose, "counts": counts, "rms": rms}
    if s.kind == "reduce":
        kf.kf_reduce_noalloc(s.fv.data_ptr(), s.K[0], s.K[1], s.mv.data_ptr(), s.mn.data_ptr(), s.K, s.pose,
                             s.model_pose, 0.16, 512, 0, s.khi, s.sums.data_ptr(), s.stream)
        return {"sums": s.sums}
    if s.kind == "map":
        kf.kf_volume_integrate(s.volume, s.depth.data_ptr(), s.K, s.pose, True)
        kf.kf_volume_raycast(s.volume, s.K, s.pose, RAY[0], RAY[1], s.dz, s.V.data_ptr(), s.N.data_ptr(), True)
        return {"vertex": s.V, "normal": s.N}
    t = s.trackers[0]
    kf.kf_set_frame(t, s.depth.data_ptr(), s.K, kf.KF_FRAME_DEVICE)
    status, pose, res = kf.kf_align(t, s.prior, s.init, s.lam)
    kf.kf_volume_raycast(s.volume, s.K, pose, RAY[0], RAY[1], s.dz, s.V.data_ptr(), s.N.data_ptr(), True)
    kf.kf_set_model(t, s.V.data_ptr(), s.N.data_ptr(), pose, s.K, True)
    counts, rms = _results([res])
    return {"status": status, "pose": pose, "counts": counts, "rms": rms, "vertex": s.V, "normal": s.N}


# ---------------------------------------------------------------------------
# the work of a pass
# ---------------------------------------------------------------------------
def _pyramid(w, h, levels):
    return [(w >> l) * (h >> l) for l in range(levels)]


def _track_work(px, levels, elem, least_iters):
    """Bytes and operations of frames of px (list of per-level pixel counts): the depth read
    once, the model maps read once; per filtered pixel 25 taps of 8 operations, per pixel of a
    map 60, per pixel and iteration 130 (transform 36, projection and distance 26, row 20,
    sums 58 of which the matched share)."""
    flops = px[0] * 200 + sum(px) * 60 + sum(p * it * 130 for p, it in zip(px, least_iters))
    return px[0] * 4 + px[0] * 6 * elem, flops


def work(case):
    c = case
    if c["kind"] == "track":
        # a level ends at the earliest after three equal medians; the original loop runs its caps
        iters = _caps(c) if c["mode"] == "original" else (3,) * c["levels"]
        b = f = 0
        for w, h in _sizes(c):
            x, y = _track_work(_pyramid(w, h, c["levels"]), c["levels"], 2 if c["fp16"] else 4, iters)
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    px = c["width"] * c["height"]
    if c["kind"] == "reduce":
        return {"bytes": 36 * px, "flops": 130 * px}
    # voxels between the camera and the surfaces, about 2.7 m away: depth^3 / 3 of the field of view
    voxel = 6.0 / c["res"]
    seen = 2.7 ** 3 / 3 * (640 / 525.0) * (c["height"] / c["width"] * 640 / 525.0) / voxel ** 3
    if c["kind"] == "map":
        return {"bytes": 16 * seen + 28 * px, "flops": 40 * seen + 400 * px}
    x, y = _track_work(_pyramid(c["width"], c["height"], 3), 3, 4, (3, 3, 3))
    return {"bytes": x + 24 * px, "flops": y + 400 * px}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _fma(a, b, c):
    """float32 a b + c rounded once (the product is exact in float64)."""
    return (a.to(F64) * (b.to(F64) if torch.is_tensor(b) else b) + (c.to(F64) if torch.is_tensor(c) else c)).to(F32)


def _rows32(R, t, v):
    """float32 rows of R v + t as chains of fused multiply-adds; R, t numpy float32."""
    return [_fma(v[2], float(R[i, 2]), _fma(v[1], float(R[i, 1]), _fma(v[0], float(R[i, 0]), float(t[i]))))
            for i in range(3)]


def _bilateral(D, radius=2, ss=4.0, sr=0.03):
    D = D.to(F64)
    ok = torch.isfinite(D) & (D > 0)
    z = torch.where(ok, D, torch.zeros_like(D))
    h, w = z.shape
    P = torch.nn.functional.pad(z, (radius,) * 4)
    num, den = torch.zeros_like(z), torch.zeros_like(z)
    for dy in range(2 * radius + 1):
        for dx in range(2 * radius + 1):
            n = P[dy:dy + h, dx:dx + w]
            e = -((dx - radius) ** 2 + (dy - radius) ** 2) / (2 * ss * ss) - (n - z) ** 2 / (2 * sr * sr)
            wt = torch.where(ok & (n > 0), torch.exp(e), torch.zeros_like(z))
            num, den = num + wt * n, den + wt
    return torch.where(ok, num / torch.where(ok, den, torch.ones_like(den)), torch.zeros_like(z))


def _half(D, sr=0.03):
    h, w = D.shape[0] // 2, D.shape[1] // 2
    blk = [D[y:2 * h:2, x:2 * w:2] for y in (0, 1) for x in (0, 1)]
    anchor = torch.zeros((h, w), device=D.device, dtype=F64)
    for b in blk:
        anchor = torch.where((anchor == 0) & (b > 0), b, anchor)
    s, n = torch.zeros_like(anchor), torch.zeros_like(anchor)
    thr = float(np.float32(3.0 * sr))
    for b in blk:
        use = (b > 0) & ((b.to(F32) - anchor.to(F32)).abs() <= thr)
        s, n = s + torch.where(use, b, torch.zeros_like(b)), n + use
    return torch.where(n > 0, s / n.clamp(min=1), torch.zeros_like(s))


def _frame_maps(D, K):
    """Vertices (float64) and normals of a level's depth; a vertex takes part when both exist."""
    w, h, fx, fy, cx, cy = K
    u = torch.arange(w, device=D.device, dtype=F64)[None, :]
    v = torch.arange(h, device=D.device, dtype=F64)[:, None]
    V = torch.stack([(u - cx) * D / fx, (v - cy) * D / fy, D], -1)
    V[~(D > 0)] = NAN
    z = D.to(F32)
    f32 = np.float32
    ix, iy = float(f32(1) / f32(fx)), float(f32(1) / f32(fy))
    V32 = torch.stack([((u.to(F32) - float(f32(cx))) * z) * ix, ((v.to(F32) - float(f32(cy))) * z) * iy, z], -1)
    V32[~(z > 0)] = NAN
    c, a, b = V32[:-1, :-1], V32[:-1, 1:] - V32[:-1, :-1], V32[1:, :-1] - V32[:-1, :-1]
    x = [a[..., i] * b[..., j] - a[..., j] * b[..., i] for i, j in ((1, 2), (2, 0), (0, 1))]
    l2 = (x[0] * x[0] + x[1] * x[1]) + x[2] * x[2]
    sd = (x[0] * c[..., 0] + x[1] * c[..., 1]) + x[2] * c[..., 2]
    ok = torch.isfinite(l2) & (l2 > 0)
    cr = torch.linalg.cross(V[:-1, 1:] - V[:-1, :-1], V[1:, :-1] - V[:-1, :-1])
    n = cr / torch.linalg.vector_norm(cr, dim=-1, keepdim=True)
    n = torch.where((sd > 0)[..., None], -n, n)
    n[~ok] = NAN
    N = torch.full_like(V, NAN)
    N[:-1, :-1] = n
    return V, N, torch.isfinite(V).all(-1) & torch.isfinite(N).all(-1)


def _matches(V, N, ok, mv, mn, mK, T, Tm, d_max, bins, cos_min=None):
    """float32 decisions: matched model pixel and distance bin per frame pixel (-1: none)."""
    f32 = np.float32
    mw, mh, fx, fy, cx, cy = mK
    Rr, tr = Tm[:3, :3].T @ T[:3, :3], Tm[:3, :3].T @ (T[:3, 3] - Tm[:3, 3])
    Rw, tw = T[:3, :3].astype(f32), T[:3, 3].astype(f32)
    v = [V[..., a].to(F32) for a in range(3)]
    m = _rows32(Rr.astype(f32), tr.astype(f32), v)
    p = _rows32(Rw, tw, v)
    rz = 1.0 / m[2]
    ur = torch.round(_fma(m[0] * float(f32(fx)), rz, float(f32(cx))))
    vr = torch.round(_fma(m[1] * float(f32(fy)), rz, float(f32(cy))))
    ok = ok & (m[2] > 0) & (ur >= 0) & (ur <= mw - 1) & (vr >= 0) & (vr <= mh - 1)
    j = torch.where(ok, vr, torch.zeros_like(vr)).long() * mw + torch.where(ok, ur, torch.zeros_like(ur)).long()
    q, nq = mv.reshape(-1, 3)[j], mn.reshape(-1, 3)[j]
    ok = ok & torch.isfinite(q).all(-1) & torch.isfinite(nq).all(-1) & (nq != 0).any(-1)
    q32 = q.to(F32)
    d = [p[a] - q32[..., a] for a in range(3)]
    dist = torch.sqrt(_fma(d[2], d[2], _fma(d[1], d[1], d[0] * d[0])))
    ok = ok & (dist < float(f32(d_max)))
    if cos_min is not None:
        n = _rows32(Rw, np.zeros(3, f32), [N[..., a].to(F32) for a in range(3)])
        n32 = nq.to(F32)
        ok = ok & ((n[0] * n32[..., 0] + n[1] * n32[..., 1]) + n[2] * n32[..., 2] >= float(f32(cos_min)))
    k = torch.floor(dist * float(f32(bins / d_max))).clamp(max=bins - 1)
    return torch.where(ok, k, torch.full_like(k, -1)).long(), q.to(F64), nq.to(F64)


def _normal_sums(V, q, n, use, T):
    """A^T A, A^T b, the pairs and sum b^2 of the point-to-plane rows of the pixels in use."""
    R = torch.from_numpy(T[:3, :3].copy()).to(V.device)
    t = torch.from_numpy(T[:3, 3].copy()).to(V.device)
    p, q, n = V[use].to(F64) @ R.T + t, q[use], n[use]
    A = torch.cat([torch.linalg.cross(p, n), n], -1)
    b = ((q - p) * n).sum(-1)
    return A.T @ A, A.T @ b, int(use.sum()), float((b * b).sum())


def _exp(w):
    t = float(np.linalg.norm(w))
    if t < 1e-12:
        return np.eye(3)
    K = np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
    return np.eye(3) + math.sin(t) / t * K + (1 - math.cos(t)) / (t * t) * (K @ K)


def _align(depth, mv, mn, K, Tm, prior, init, lam, levels, caps, original=False):
    """Pose and rms residual of the coarse-to-fine alignment in 64 bits."""
    bins, d_max = 512, 0.16
    D, T = _bilateral(depth), init.copy()
    if not original:
        T[:3, :3] = prior
    fk, mk, frame, model = K, K, [], []
    for l in range(levels):
        if l:
            D, mv, mn = _half(D), mv[:mk[1] // 2 * 2:2, :mk[0] // 2 * 2:2], mn[:mk[1] // 2 * 2:2, :mk[0] // 2 * 2:2]
            fk = (fk[0] // 2, fk[1] // 2, fk[2] / 2, fk[3] / 2, (fk[4] - 0.5) / 2, (fk[5] - 0.5) / 2)
            mk = (mk[0] // 2, mk[1] // 2, mk[2] / 2, mk[3] / 2, mk[4] / 2, mk[5] / 2)
        frame.append(_frame_maps(D, fk))
        model.append((mv, mn, mk))
    cos_min = math.cos(math.radians(20.0)) if original else None
    rms = 0.0
    for l in reversed(range(levels)):
        medians = []
        for _ in range(caps[l]):
            V, N, ok = frame[l]
            k, q, n = _matches(V, N, ok, *model[l], T, Tm, d_max, bins, cos_min)
            hist = torch.bincount(k[k >= 0], minlength=bins).cpu().numpy()
            if hist.sum() < 6:
                return T, rms
            med = int(np.argmax(2 * np.cumsum(hist) >= hist.sum()))
            khi = bins - 1 if original else min(bins - 1, 2 * med + 1)
            use = (k >= 0) & (k <= khi)
            H, g, cnt, sb2 = _normal_sums(V, q, n, use, T)
            if cnt < 6:
                return T, rms
            H, g = H.cpu().numpy(), g.cpu().numpy()
            H[:3, :3] += 2 * lam * cnt * np.eye(3)
            x = np.linalg.solve(H, g)
            T = _pose(_exp(x[:3]), x[3:]) @ T
            rms = math.sqrt(sb2 / cnt)
            medians.append(med)
            if not original and len(medians) >= 3 and len(set(medians[-3:])) == 1:
                break
    return T, rms


def _row(R, t, x, y, z):
    """((R0 x + R1 y) + R2 z) + t, each operation rounded to float32."""
    return ((float(R[0]) * x + float(R[1]) * y) + float(R[2]) * z) + float(t)


class _Field:
    """The volume as plain float32 arrays, every operation rounded once, as the library states it."""

    def __init__(self, vp):
        f32 = np.float32
        self.res, self.s = vp.res, float(f32(vp.side) / f32(vp.res))
        self.o, self.mu, self.w_max = [float(v) for v in vp.origin], float(f32(vp.mu)), vp.w_max
        self.F = torch.ones((vp.res,) * 3, device="cuda", dtype=F32)
        self.W = torch.zeros((vp.res,) * 3, device="cuda", dtype=F32)

    def integrate(self, D, K, T):
        f32 = np.float32
        Rt = T[:3, :3].T.astype(f32)
        tt = (-(T[:3, :3].T @ T[:3, 3])).astype(f32)
        w, h, fx, fy, cx, cy = K
        idx = torch.arange(self.res, device="cuda", dtype=F32) + 0.5
        x, y = (idx * self.s + self.o[0])[None, None, :], (idx * self.s + self.o[1])[None, :, None]
        for a in range(0, self.res, 64):
            part = slice(a, min(self.res, a + 64))
            z = (idx[part] * self.s + self.o[2])[:, None, None]
            px, py, pz = (_row(Rt[i], tt[i], x, y, z) for i in range(3))
            ur = torch.round((px * float(f32(fx))) / pz + float(f32(cx)))
            vr = torch.round((py * float(f32(fy))) / pz + float(f32(cy)))
            ok = (pz > 0) & (ur >= 0) & (ur <= w - 1) & (vr >= 0) & (vr <= h - 1)
            j = torch.where(ok, vr, torch.zeros_like(vr)).long() * w + torch.where(ok, ur, torch.zeros_like(ur)).long()
            d = D.reshape(-1)[j]
            eta = d - pz
            ok = ok & torch.isfinite(d) & (d > 0) & (eta >= -self.mu)
            mu = torch.tensor(self.mu, device="cuda", dtype=F32)
            f = (eta / mu).clamp(max=1.0)
            F, W = self.F[part], self.W[part]
            self.F[part] = torch.where(ok, (W * F + f) / (W + 1), F)
            self.W[part] = torch.where(ok, (W + 1).clamp(max=self.w_max), W)

    def sample(self, q):
        """Trilinear value and whether all eight corners were observed."""
        s = torch.tensor(self.s, device="cuda", dtype=F32)
        g = [(q[a] - self.o[a]) / s - 0.5 for a in range(3)]
        f = [torch.floor(x) for x in g]
        ok = torch.ones_like(f[0], dtype=torch.bool)
        for x in f:
            ok = ok & (x >= 0) & (x <= self.res - 2)
        t = [a - b for a, b in zip(g, f)]
        i = [torch.where(ok, x, torch.zeros_like(x)).long() for x in f]
        b = (i[2] * self.res + i[1]) * self.res + i[0]
        c = []
        for dz in (0, 1):
            for dy in (0, 1):
                for dx in (0, 1):
                    j = b + ((dz * self.res + dy) * self.res + dx)
                    ok = ok & (self.W.reshape(-1)[j] > 0)
                    c.append(self.F.reshape(-1)[j])
        mix = lambda p, r, u: p + u * (r - p)  # noqa: E731
        lo = mix(mix(c[0], c[1], t[0]), mix(c[2], c[3], t[0]), t[1])
        hi = mix(mix(c[4], c[5], t[0]), mix(c[6], c[7], t[0]), t[1])
        return mix(lo, hi, t[2]), ok

    def raycast(self, K, T, zn, zf, dz):
        f32 = np.float32
        w, h, fx, fy, cx, cy = K
        R, c = T[:3, :3].astype(f32), T[:3, 3].astype(f32)
        one = torch.ones((h, w), device="cuda", dtype=F32)
        fx, fy = (torch.tensor(float(f32(v)), device="cuda", dtype=F32) for v in (fx, fy))
        dx = ((torch.arange(w, device="cuda", dtype=F32) - float(f32(cx))) / fx)[None, :] * one
        dy = ((torch.arange(h, device="cuda", dtype=F32) - float(f32(cy))) / fy)[:, None] * one
        d = [_row(R[a], 0.0, dx, dy, one) for a in range(3)]
        at = lambda z: [float(c[a]) + z * d[a] for a in range(3)]  # noqa: E731
        live, have = torch.ones_like(one, dtype=torch.bool), torch.zeros_like(one, dtype=torch.bool)
        hit, zp, fp, zs = torch.zeros_like(have), torch.zeros_like(one), torch.zeros_like(one), torch.zeros_like(one)
        zn, zf, dz = f32(zn), f32(zf), f32(dz)
        k = 0
        while (z := f32(zn + f32(f32(k) * dz))) <= zf:
            k += 1
            f, ok = self.sample(at(float(z)))
            cross = live & ok & have & (fp > 0) & (f <= 0)
            back = live & ok & have & (fp < 0) & (f > 0)
            zs = torch.where(cross, zp + float(dz) * (fp / (fp - f)), zs)
            hit, live = hit | cross, live & ~(cross | back)
            have, zp, fp = ok, torch.where(ok, torch.full_like(zp, float(z)), zp), torch.where(ok, f, fp)
        v = at(zs)
        g = []
        for a in range(3):
            side = []
            for step in (self.s, -self.s):
                q = list(v)
                q[a] = q[a] + step
                f, ok = self.sample(q)
                hit = hit & ok
                side.append(f.to(F64))
            g.append(side[0] - side[1])
        g = torch.stack(g, -1)
        ln = torch.linalg.vector_norm(g, dim=-1, keepdim=True)
        hit = (hit & (ln[..., 0] > 0))[..., None]
        nan = torch.full_like(g, NAN)
        return torch.where(hit, torch.stack(v, -1).to(F64), nan), torch.where(hit, g / ln, nan)


def exact(case, seed):
    c = case
    if c["kind"] == "track":
        if c["mode"] == "shooting":
            return None  # 25 candidates a pixel and iteration: longer than a check should take
        got = [_align(p["depth"], p["mv"], p["mn"], p["K"], p["base"], p["prior"], p["base"], c["lam"], c["levels"],
                      _caps(c), c["mode"] == "original") for p in _pairs(c, seed)]
        pose, rms = np.stack([g[0] for g in got]), np.array([g[1] for g in got])
        return {"status": None, "pose": pose[0] if len(got) == 1 else pose, "counts": None, "rms": rms}
    if c["kind"] == "reduce":
        s = _prepare_reduce(c, seed)
        ok = torch.isfinite(s.fv).all(-1)
        k, q, n = _matches(s.fv, None, ok, s.mv, s.mn, s.K, s.pose, s.model_pose, 0.16, 512)
        H, g, cnt, sb2 = _normal_sums(s.fv, q, n, (k >= 0) & (k <= s.khi), s.pose)
        iu = torch.triu_indices(6, 6)
        tail = torch.tensor([float(cnt), sb2], dtype=F64, device="cuda")
        return {"sums": torch.cat([H[iu[0], iu[1]], g, tail])}
    vp, K, path, depths = _walk(c, seed)
    field = _Field(vp)
    for D, T in zip(depths[:-1], path[:-1]):
        field.integrate(D, K, T)
    if c["kind"] == "map":
        field.integrate(depths[-1], K, path[-1])
        V, N = field.raycast(K, path[-1], RAY[0], RAY[1], _step(vp))
        return {"vertex": V, "normal": N}
    V, N = field.raycast(K, path[-2], RAY[0], RAY[1], _step(vp))
    pose, rms = _align(depths[-1], V.to(F32), N.to(F32), K, path[-2], path[-1][:3, :3], path[-2], 5.0, 3, (10, 5, 4))
    V, N = field.raycast(K, pose, RAY[0], RAY[1], _step(vp))
    return {"status": None, "pose": pose, "counts": None, "rms": np.array([rms]), "vertex": V, "normal": N}
