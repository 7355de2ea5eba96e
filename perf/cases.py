"""The calls that users of pl3d make, as measurable cases: single organized frames from small to
large, odd sizes with every optional output, larger windows, batches, host-buffer frames, and the
two consumers of the results (explicit mesh with segment lists, Gaussian accumulator).

Inputs are seeded synthetic scans made on the GPU: a pinhole depth camera in a room corner (floor,
two walls, boxes, on larger frames a ramp and outliers) and a spinning LiDAR on a street (road,
sidewalks, facades, cars), ray-cast in FP64, with range noise and missing returns, as FP32 xyz.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2007_12065_gb300 as pl3d

DEV = "cuda"
MIXED_SIZES = [(120, 160), (240, 320), (480, 640), (64, 1024), (128, 2048)]
LIDAR_SHAPE = 6          # an aspect ratio from which a scan is a spinning LiDAR's
FASTGA_LEVEL = 4


# ------------------------------------------------------------------------------- the cases


def _frame(H, W, **kw):
    c = dict(kind="frame", H=H, W=W, lap=5, bil=3, lap_kernel=3, bil_kernel=3, extras=False, min_triangles=0,
             max_offset=0.0)
    c.update(kw)
    return c


def listed():
    return [
        # a small depth camera, one call per frame from the convenience wrapper: launches and latency
        _frame(120, 160, name="depth_120x160", kind="wrapper"),
        # the ordinary frame of a depth camera, outputs kept by the caller
        _frame(480, 640, name="depth_480x640"),
        # the largest sensor of the served mix
        _frame(720, 1280, name="depth_720x1280"),
        # a spinning LiDAR scan: few rows, many columns, its own iteration counts
        _frame(64, 1024, name="lidar_64x1024", lap=3, bil=2),
        # odd sizes (no 16-byte rows), smoothed points and groups exported, small segments dropped and
        # the plane-offset test on
        _frame(243, 317, name="ragged_243x317_options", lap=2, bil=2, extras=True, min_triangles=25, max_offset=0.02),
        # the synthetic benchmark of the paper: 500 x 500 points, Laplacian window 5; bilateral window 5 too
        _frame(500, 500, name="windows5_500x500", lap=2, bil=2, lap_kernel=5, bil_kernel=5),
        # 256 frames of mixed sizes in one launch
        dict(name="batch_256_mixed", kind="batch", n=256, lap=5, bil=3, lidar_lap=3, lidar_bil=2, extras=False),
        # one iteration of each filter over a batch, smoothed points exported
        dict(name="batch_64_one_iteration", kind="batch", n=64, lap=1, bil=1, lidar_lap=1, lidar_bil=1, extras=True),
        # explicit mesh and segment lists of a frame, the input of polygon extraction
        dict(name="mesh_480x640", kind="mesh", H=480, W=640),
        # dominant normals from a frame's triangle normals
        dict(name="fastga_480x640", kind="fastga", H=480, W=640, stride=1),
        # a stream of frames from page-locked host buffers
        dict(name="stream_6x480x640", kind="stream", H=480, W=640, n=6, lap=5, bil=3),
        # one lone frame from page-locked host buffers: the latency of a synchronous call
        dict(name="host_240x320", kind="host", H=240, W=320, lap=5, bil=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    def depth_size(most=720 * 1280):
        while True:
            H = _log_int(rng, 100, 720)
            W = int(H * rng.uniform(1.0, 1.8))
            if rng.random() < 0.5:
                H, W = H & ~3, W & ~3
            if H * W <= most:
                return H, W

    kind = rng.choice(["frame", "frame", "frame", "wrapper", "lidar", "lidar", "options", "windows", "batch",
                       "batch", "mesh", "fastga", "stream", "host"])
    if kind in ("frame", "wrapper"):
        H, W = depth_size()
        return _frame(H, W, kind=kind, lap=rng.randint(2, 6), bil=rng.randint(1, 4))
    if kind == "lidar":
        H, W = _log_int(rng, 32, 128), rng.choice([1024, 1800, 2048, rng.randint(900, 2048)])
        return _frame(H, W, lap=rng.randint(2, 4), bil=rng.randint(1, 3))
    if kind == "options":
        H, W = depth_size(480 * 640)
        return _frame(H, W, lap=rng.randint(1, 5), bil=rng.randint(1, 3), extras=True,
                      min_triangles=rng.randint(1, 60), max_offset=rng.choice([0.0, 0.02, 0.05]))
    if kind == "windows":
        H, W = depth_size(500 * 500)
        return _frame(H, W, lap=rng.randint(1, 2), bil=rng.randint(1, 2), lap_kernel=rng.choice([3, 5]),
                      bil_kernel=rng.choice([3, 5]))
    if kind == "batch":
        one = rng.random() < 0.3
        lap, bil = (1, 1) if one else (rng.randint(2, 5), rng.randint(1, 3))
        return dict(kind="batch", n=_log_int(rng, 8, 200), lap=lap, bil=bil, lidar_lap=min(lap, 3),
                    lidar_bil=min(bil, 2), extras=one, pick=rng.randint(0, 999))
    H, W = depth_size(480 * 640)
    if kind == "mesh":
        return dict(kind="mesh", H=H, W=W)
    if kind == "fastga":
        return dict(kind="fastga", H=H, W=W, stride=rng.choice([1, 1, 2, 3]))
    if kind == "stream":
        return dict(kind="stream", H=H, W=W, n=rng.randint(3, 6), lap=rng.randint(2, 5), bil=rng.randint(1, 3))
    return dict(kind="host", H=H, W=W, lap=rng.randint(2, 5), bil=rng.randint(1, 3))


# ------------------------------------------------------------------------------- the scans


def _is_lidar(H, W):
    return W >= LIDAR_SHAPE * H


def _cast(d, o, planes, boxes):
    """Nearest positive hit distance of rays o + t d [P, 3] against axis-aligned patches (axis,
    value, {other axis: (lo, hi)}) and boxes [K, 2, 3]; inf without one."""
    t_best = torch.full(d.shape[:1], math.inf, dtype=torch.float64, device=DEV)
    for axis, value, bounds in planes:
        t = (value - o[axis]) / d[:, axis]
        ok = t > 1e-9
        for a, (lo, hi) in bounds.items():
            p = o[a] + t * d[:, a]
            ok &= (p >= lo) & (p <= hi)
        t_best = torch.where(ok & (t < t_best), t, t_best)
    if boxes:
        b = torch.tensor(boxes, dtype=torch.float64, device=DEV)               # [K, 2, 3]
        org = torch.tensor(o, dtype=torch.float64, device=DEV)
        t0 = (b[:, None, 0] - org) / d[None]
        t1 = (b[:, None, 1] - org) / d[None]
        near, far = torch.minimum(t0, t1).amax(-1), torch.maximum(t0, t1).amin(-1)
        t = torch.where((far >= near) & (near > 1e-9), near, math.inf).amin(0)
        t_best = torch.minimum(t_best, t)
    return t_best


def _depth_scene(H, W, rnd):
    yaw, pitch = math.radians(45.0), math.radians(30.0)
    f = np.array([math.cos(yaw) * math.cos(pitch), math.sin(yaw) * math.cos(pitch), -math.sin(pitch)])
    r = np.array([math.sin(yaw), -math.cos(yaw), 0.0])
    dn = np.cross(f, r)
    fx = (W / 2.0) / math.tan(math.radians(70.0) / 2.0)
    u = (torch.arange(H, dtype=torch.float64, device=DEV) - (H - 1) / 2.0) / fx
    v = (torch.arange(W, dtype=torch.float64, device=DEV) - (W - 1) / 2.0) / fx
    vec = lambda a: torch.tensor(a, dtype=torch.float64, device=DEV)  # noqa: E731
    d = u[:, None, None] * vec(dn) + v[None, :, None] * vec(r) + vec(f)
    d = (d / d.norm(dim=-1, keepdim=True)).reshape(-1, 3)
    big = H * W >= 300 * 400
    boxes = []
    for _ in range(12 if big else 4):
        sx, sy, sz = (rnd.uniform(0.2, 0.6) for _ in range(3))
        x, y = rnd.uniform(0.6, 2.6), rnd.uniform(0.6, 2.6)
        boxes.append([[x - sx / 2, y - sy / 2, 0.0], [x + sx / 2, y + sy / 2, sz]])
    o = (0.0, 0.0, 1.5)
    t = _cast(d, o, [(2, 0.0, {}), (0, 3.0, {}), (1, 3.0, {})], boxes)
    dominant = [[0, 0, 1], [-1, 0, 0], [0, -1, 0]]
    if big:
        # a 1.2 m x 0.8 m ramp rising away from the camera at 15 degrees
        ang, s0 = math.radians(15.0), rnd.uniform(1.3, 1.8)
        hz = np.array([math.cos(yaw), math.sin(yaw), 0.0])
        a = math.cos(ang) * hz + np.array([0.0, 0.0, math.sin(ang)])
        b = np.array([-math.sin(yaw), math.cos(yaw), 0.0])
        n = np.cross(a, b)
        n = n if n[2] > 0 else -n
        p0 = np.array([s0 * hz[0], s0 * hz[1], 0.002])
        tr = float((p0 - np.array(o)) @ n) / (d @ vec(n))
        p = vec(o) + tr[:, None] * d - vec(p0)
        along, across = p @ vec(a), p @ vec(b)
        ok = (tr > 0) & (along >= 0) & (along <= 1.2) & (across.abs() <= 0.4) & (tr < t)
        t = torch.where(ok, tr, t)
        dominant.append([float(x) for x in n])
    return d, o, t, dominant, dict(sigma=0.005, outliers=0.01 if big else 0.0, missing=0.03 if big else 0.02,
                                   reach=math.inf)


def _lidar_scene(H, W, rnd):
    el = torch.linspace(math.radians(3.0), math.radians(-25.0), H, dtype=torch.float64, device=DEV)[:, None]
    az = (math.pi - torch.arange(W, dtype=torch.float64, device=DEV) * (2 * math.pi / W))[None, :]
    d = torch.stack([el.cos() * az.cos(), el.cos() * az.sin(), el.sin().expand(H, W)], -1).reshape(-1, 3)
    planes = [(2, 0.0, {1: (-4.0, 4.0)})]
    for s in (1.0, -1.0):
        planes += [(2, 0.15, {1: (min(4.0 * s, 10.0 * s), max(4.0 * s, 10.0 * s))}), (1, 4.0 * s, {2: (0.0, 0.15)}),
                   (1, 10.0 * s, {2: (0.0, 15.0)})]
    boxes = []
    while len(boxes) < 20:
        x, y = rnd.uniform(-60, 60), rnd.uniform(-3, 3)
        if abs(x) > 6:
            boxes.append([[x - 2.25, y - 0.9, 0.0], [x + 2.25, y + 0.9, 1.5]])
    o = (0.0, 0.0, 1.8)
    return d, o, _cast(d, o, planes, boxes), [[0, 0, 1], [0, -1, 0]], dict(sigma=0.02, outliers=0.0, missing=0.10,
                                                                           reach=100.0)


def _scans(H, W, n, seed):
    """n scans of one scene: points float32 [n, H, W, 3] (NaN = missing) and the dominant normals."""
    rnd = random.Random(seed * 7919 + H * 31 + W)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(rnd.getrandbits(48))
    d, o, t, dominant, noise = (_lidar_scene if _is_lidar(H, W) else _depth_scene)(H, W, rnd)
    shape = (n, H * W)
    tn = t + noise["sigma"] * torch.randn(shape, dtype=torch.float64, device=DEV, generator=gen)
    if noise["outliers"] > 0:
        hit = torch.rand(shape, device=DEV, generator=gen) < noise["outliers"]
        tn += hit * (0.6 * torch.rand(shape, dtype=torch.float64, device=DEV, generator=gen) - 0.3)
    ok = torch.isfinite(t) & (tn > 0) & (tn <= noise["reach"])
    ok &= torch.rand(shape, device=DEV, generator=gen) >= noise["missing"]
    p = torch.where(ok, tn, math.nan)[..., None] * d + torch.tensor(o, dtype=torch.float64, device=DEV)
    return p.to(torch.float32).reshape(n, H, W, 3), np.array(dominant, np.float32)


def _params(case, H, W):
    lidar = _is_lidar(H, W)
    lap, bil = case.get("lap", 5), case.get("bil", 3)
    if lidar and "lidar_lap" in case:
        lap, bil = case["lidar_lap"], case["lidar_bil"]
    return dict(lap_iters=lap, lap_lambda=1.0, lap_kernel=case.get("lap_kernel", 3), bil_iters=bil,
                bil_sigma_len=0.1, bil_sigma_ang=0.15, bil_kernel=case.get("bil_kernel", 3),
                max_edge=0.5 if lidar else 0.1, min_dot=0.95, max_offset=case.get("max_offset", 0.0),
                min_triangles=case.get("min_triangles", 0))


def _batch_sizes(case):
    """Sizes of a batch's frames, in its order: the same for every seed, so that the work is too."""
    rnd = random.Random(104 + case.get("pick", 0))
    return [rnd.choice(MIXED_SIZES) for _ in range(case["n"])]


# ------------------------------------------------------------------------------- what a program keeps

_kept: dict = {}


def _extractor():
    """The program's one extractor (its context keeps the scratch)."""
    if "extractor" not in _kept:
        _kept["extractor"] = pl3d.PlaneExtractor(0)
    return _kept["extractor"]


def _pipeline(points):
    if _kept.get("pipeline", (0, 0))[1] < points:
        if "pipeline" in _kept:
            pl3d.pl3d_pipeline_destroy(_kept["pipeline"][0])
        _kept["pipeline"] = (pl3d.pl3d_pipeline_create(0, points, 3), points)
    return _kept["pipeline"][0]


def _outputs(n, H, W, extras, device=DEV, pin=False):
    q = 2 * (H - 1) * (W - 1)
    kw = dict(device=device, pin_memory=pin)
    o = dict(mask=torch.empty((n, q), dtype=torch.uint8, **kw), normals=torch.empty((n, q, 3), dtype=torch.float32, **kw),
             labels=torch.empty((n, q), dtype=torch.int32, **kw))
    if extras:
        o["points"] = torch.empty((n, H, W, 3), dtype=torch.float32, **kw)
        o["groups"] = torch.empty((n, q), dtype=torch.uint8, **kw)
    return o


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind)
    if kind == "batch":
        sizes = _batch_sizes(case)
        scans, batch, outs = {}, pl3d.Batch(), {k: [] for k in ("mask", "normals", "labels", "points", "groups")}
        for size in sorted(set(sizes)):
            scans[size] = _scans(*size, sizes.count(size), seed)
        n_tri = [2 * (H - 1) * (W - 1) for H, W in sizes]
        n_pts = [H * W for H, W in sizes]
        big = dict(mask=torch.empty(sum(n_tri), dtype=torch.uint8, device=DEV),
                   normals=torch.empty((sum(n_tri), 3), dtype=torch.float32, device=DEV),
                   labels=torch.empty(sum(n_tri), dtype=torch.int32, device=DEV))
        if case["extras"]:
            big["points"] = torch.empty((sum(n_pts), 3), dtype=torch.float32, device=DEV)
            big["groups"] = torch.empty(sum(n_tri), dtype=torch.uint8, device=DEV)
        outs = {k: v.split(n_pts if k == "points" else n_tri) for k, v in big.items()}
        used = dict.fromkeys(scans, 0)
        for i, size in enumerate(sizes):
            pts, nd = scans[size]
            batch.add(pts[used[size]], *size, pl3d.make_params(**_params(case, *size)), nd, outs["mask"][i],
                      outs["normals"][i], outs["labels"][i], outs["points"][i] if case["extras"] else None,
                      outs["groups"][i] if case["extras"] else None)
            used[size] += 1
        s.update(ctx=_extractor().ctx, batch=batch, out=big)
        return s
    H, W, n = case["H"], case["W"], case.get("n", 1)
    pts, nd = _scans(H, W, n, seed)
    s.update(H=H, W=W, n=n, nd=nd, params=pl3d.make_params(**_params(case, H, W)))
    if kind in ("stream", "host"):
        s["points"] = torch.empty(pts.shape, dtype=torch.float32, pin_memory=True)
        s["points"].copy_(pts)
        s["out"] = _outputs(n, H, W, False, "cpu", True)
        s["handle"] = _pipeline(H * W) if kind == "stream" else _extractor().ctx
        s["frames"] = [dict(points=s["points"][i], **{k: v[i] for k, v in s["out"].items()}) for i in range(n)]
        return s
    s["points"] = pts[0]
    s["extractor"], s["ctx"] = _extractor(), _extractor().ctx
    q = 2 * (H - 1) * (W - 1)
    if kind == "frame":
        s["out"] = {k: v[0] for k, v in _outputs(1, H, W, case["extras"]).items()}
    elif kind == "mesh":
        s["labels"] = _extractor()(pts[0], s["params"], nd)["labels"]
        sizes = dict(T=3 * q, Tmap=q, HE=3 * q, seg_labels=q, seg_offsets=q + 1, seg_tris=q)
        # only the first counts[...] entries are written: the rest keep this value
        s["out"] = {k: torch.full((v,), -1, dtype=torch.int32, device=DEV) for k, v in sizes.items()}
        s["out"]["counts"] = torch.zeros(3, dtype=torch.int64, device=DEV)
        s["out"]["border"] = torch.zeros(q, dtype=torch.uint8, device=DEV)
    elif kind == "fastga":
        out = _extractor()(pts[0], s["params"], nd)
        s.update(normals=out["normals"], mask=out["mask"], stride=case["stride"])
        s["out"] = dict(counts=torch.empty(20 * 4 ** FASTGA_LEVEL, dtype=torch.int32, device=DEV))
    return s


def run(s):
    kind = s["kind"]
    if kind == "wrapper":
        return s["extractor"](s["points"], s["params"], s["nd"])
    o = s["out"]
    if kind == "frame":
        pl3d.pl3d_extract_planes_ex(s["ctx"], s["points"], s["H"], s["W"], s["params"], s["nd"], len(s["nd"]), o["mask"],
                                    o["normals"], o["labels"], o.get("points"), o.get("groups"))
    elif kind == "batch":
        pl3d.pl3d_extract_planes_batched(s["ctx"], s["batch"])
    elif kind == "mesh":
        pl3d.pl3d_extract_mesh(s["ctx"], s["points"], s["labels"], s["H"], s["W"], o["T"], o["Tmap"], o["HE"], o["counts"],
                               o["seg_labels"], o["seg_offsets"], o["seg_tris"], o["border"])
    elif kind == "fastga":
        pl3d.pl3d_fastga(s["ctx"], s["normals"], s["mask"], s["mask"].numel(), FASTGA_LEVEL, s["stride"], o["counts"])
    elif kind == "stream":
        tickets = [pl3d.pl3d_pipeline_submit(s["handle"], f["points"], s["H"], s["W"], s["params"], s["nd"], len(s["nd"]),
                                             f["mask"], f["normals"], f["labels"]) for f in s["frames"]]
        for t in tickets:
            pl3d.pl3d_pipeline_wait(s["handle"], t)
    else:
        f = s["frames"][0]
        pl3d.pl3d_extract_planes_host(s["handle"], f["points"], s["H"], s["W"], s["params"], s["nd"], len(s["nd"]),
                                      f["mask"], f["normals"], f["labels"])
    return o


# ------------------------------------------------------------------------------- work


def _frame_work(H, W, p, K, extras):
    """Bytes and FLOP (an FMA counts two, an exponential or a root one) of one frame: points in,
    normals, mask and labels out; per point, iteration and neighbour 16; per triangle, iteration and
    window triangle 26; per triangle 30 for its geometry and 5 per dominant normal."""
    npx, q = H * W, 2 * (H - 1) * (W - 1)
    by = 12 * npx + 17 * q + ((12 * npx + q) if extras else 0)
    fl = 16 * npx * p["lap_iters"] * (p["lap_kernel"] ** 2 - 1) + q * (26 * p["bil_iters"] * 2 * p["bil_kernel"] ** 2 + 30 + 5 * K)
    return by, fl


def work(case):
    kind = case["kind"]
    groups = lambda H, W: 2 if _is_lidar(H, W) else (4 if H * W >= 300 * 400 else 3)  # noqa: E731
    if kind == "batch":
        each = [_frame_work(H, W, _params(case, H, W), groups(H, W), case["extras"]) for H, W in _batch_sizes(case)]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    H, W = case["H"], case["W"]
    q = 2 * (H - 1) * (W - 1)
    if kind == "mesh":      # points and labels in; T, T_map, HE, segment lists and border bits out
        return {"bytes": 12 * H * W + 4 * q + (12 + 4 + 12 + 4 + 1) * q, "flops": 0}
    if kind == "fastga":    # 13 bytes per triangle read; its nearest cell by one dot product at least
        m = -(-q // case["stride"])
        return {"bytes": 13 * m + 4 * 20 * 4 ** FASTGA_LEVEL, "flops": 5 * m}
    b, f = _frame_work(H, W, _params(case, H, W), groups(H, W), case.get("extras", False))
    return {"bytes": b * case.get("n", 1), "flops": f * case.get("n", 1)}


# ------------------------------------------------------------------------------- 64 bits


def _laplacian64(P, ok, p):
    n, H, W, _ = P.shape
    R = p["lap_kernel"] // 2
    V = torch.where(ok[..., None], P, 0.0)
    for _ in range(p["lap_iters"]):
        c, own = V[:, R:H - R, R:W - R], ok[:, R:H - R, R:W - R]
        S, Ws = torch.zeros_like(c), torch.zeros_like(c[..., 0])
        for du in range(-R, R + 1):
            for dv in range(-R, R + 1):
                if du == 0 and dv == 0:
                    continue
                e = V[:, R + du:H - R + du, R + dv:W - R + dv] - c
                d = e.norm(dim=-1)
                w = torch.where(ok[:, R + du:H - R + du, R + dv:W - R + dv] & own & (d > 0), 1.0 / d, 0.0)
                S += w[..., None] * e
                Ws += w
        step = torch.where(Ws > 0, p["lap_lambda"] / Ws, 0.0)
        new = V.clone()
        new[:, R:H - R, R:W - R] = c + step[..., None] * S
        V = new
    return V


def _normals64(V, ok, p):
    """Filtered normals [n, 2 Q, 3] of smoothed points V, NaN where a triangle has none."""
    n, H, W, _ = V.shape
    p1, p2, p3, p4 = V[:, :-1, :-1], V[:, :-1, 1:], V[:, 1:, 1:], V[:, 1:, :-1]
    o1, o2, o3, o4 = ok[:, :-1, :-1], ok[:, :-1, 1:], ok[:, 1:, 1:], ok[:, 1:, :-1]
    cr = torch.stack([torch.linalg.cross(p2 - p3, p1 - p3), torch.linalg.cross(p4 - p1, p3 - p1)], 3)
    C = torch.stack([p3 + p2 + p1, p1 + p4 + p3], 3) / 3.0
    ln = cr.norm(dim=-1)
    has = torch.stack([o1 & o2 & o3, o1 & o3 & o4], 3) & (ln > 1e-20)
    N = torch.where(has[..., None], cr / ln[..., None], 0.0)
    R, Hq, Wq = p["bil_kernel"] // 2, H - 1, W - 1
    pad = lambda x, f: torch.nn.functional.pad(x, [0, 0] * (x.dim() - 3) + [R, R, R, R], value=f)  # noqa: E731
    Cp, hp = pad(C, 0.0), pad(has.to(torch.float64), 0.0)
    kc, ks = 0.5 / p["bil_sigma_len"] ** 2, 0.5 / p["bil_sigma_ang"] ** 2
    for _ in range(p["bil_iters"]):
        Np, S = pad(N, 0.0), torch.zeros_like(N)
        for du in range(2 * R + 1):
            for dv in range(2 * R + 1):
                for j in range(2):
                    cut = (slice(None), slice(du, du + Hq), slice(dv, dv + Wq), slice(j, j + 1))
                    nj = Np[cut]
                    w = torch.exp(-kc * (C - Cp[cut]).square().sum(-1) - ks * (N - nj).square().sum(-1)) * hp[cut]
                    S += w[..., None] * nj
        l = S.norm(dim=-1)
        N = torch.where((has & (l > 0))[..., None], S / l[..., None], N)
    return torch.where(has[..., None], N, math.nan).reshape(n, 2 * Hq * Wq, 3)


def _smooth64(pts, p, chunk=16):
    """Smoothed points and filtered normals of scans [n, H, W, 3] in 64 bits."""
    points, normals = [], []
    for part in pts.split(chunk):
        ok = (part.isfinite() & (part.abs() < 1e18)).all(-1)
        V = _laplacian64(part.to(torch.float64), ok, p)
        points.append(torch.where(ok[..., None], V, math.nan))
        normals.append(_normals64(V, ok, p))
    return torch.cat(points), torch.cat(normals)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("mesh", "fastga"):
        return None     # whole numbers only
    if kind == "batch":
        sizes, done = _batch_sizes(case), {}
        for size in sorted(set(sizes)):
            pts, _ = _scans(*size, sizes.count(size), seed)
            done[size] = [iter(x) for x in _smooth64(pts, _params(case, *size))]
        both = [[next(x) for x in done[size]] for size in sizes]
        out = dict(mask=None, normals=torch.cat([b[1] for b in both]), labels=None)
        if case["extras"]:
            out.update(points=torch.cat([b[0].reshape(-1, 3) for b in both]), groups=None)
        return out
    pts, _ = _scans(case["H"], case["W"], case.get("n", 1), seed)
    points, normals = _smooth64(pts, _params(case, case["H"], case["W"]))
    one = kind in ("frame", "wrapper")
    out = dict(mask=None, normals=normals[0] if one else normals, labels=None)
    if case.get("extras"):
        out.update(points=points[0], groups=None)
    return out
