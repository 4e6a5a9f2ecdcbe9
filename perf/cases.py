"""The work this rasterizer is used for, as measurable cases, each through its public entry points.

The scenes follow the synthetic ones of the tests and the benchmark: a 6 x 5 x 3 m room covered by
a triangle soup of 1-5 cm faces seen from a circle of poses, random triangles in front of one
camera, and an indexed height-field mesh.  The kinds of case are what a program does with the
library:

* ``frame``     one small view, call by call: forward, L1 loss, backward, pose gradient;
* ``step``      a mapping window under the plain L1 colour + depth loss, one graph replay a pass;
* ``mapping``   a mapping window under the whole mapping loss (D-SSIM, normals, equilateral term);
* ``track``     one iteration of camera tracking over several pose hypotheses, one graph replay;
* ``render``    the render requests of a serving loop on a forward-only plan;
* ``loss``      the photometric loss (L1 + D-SSIM + depth) and its image gradients alone;
* ``keyframes`` a forward with the map statistics and the views' co-visibility;
* ``mesh``      an indexed mesh with the smallest vertex opacity and per-face window exponents.

``exact`` evaluates the same mathematics in 64 bits with plain torch: every (face, pixel) pair of a
tile densely, gradients by autograd.  Its screen-space vertices are the float32 values of Eq. 1 in the
operation order the library documents: the window's slope grows without bound towards a face's edge,
so that vertices placed 1e-5 px apart give gradients that say nothing of each other's precision.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2605_31419_gb300 as ts

DEV = "cuda"
FOCAL = {"320x240": 262.5, "640x480": 525.0, "1200x680": 600.0, "256x256": 256.0}


# ---------------------------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest call: one view of a small map, launched call by call
        dict(name="frame_160x120", kind="frame", sizes="160x120", focal=150.0, views=1, faces=2000),
        # the same view as a training loop runs it: the captured step
        dict(name="step_160x120", kind="step", scene="triangles", sizes="160x120", focal=150.0, views=1, faces=2000),
        # mapping a room-scale map from a trajectory: the benchmark's batched step
        dict(name="step_room_20", kind="step", scene="room", sizes="1200x680", focal=0.0, views=20, faces=300000),
        # a mapping window of keyframes of uneven resolution on a dense map
        dict(name="step_window_12", kind="step", scene="room", sizes="320x240,640x480,1200x680", focal=0.0, views=12,
             faces=1000000),
        # a mapping window under the whole mapping loss, rendered normals included
        dict(name="mapping_6", kind="mapping", sizes="320x240,640x480,1200x680", focal=0.0, views=6, faces=300000),
        # tracking: many hypotheses of one frame under the D-SSIM tracking loss
        dict(name="track_64", kind="track", sizes="640x480", focal=0.0, views=64, faces=150000, ssim=0.2),
        # tracking on a small device-bound budget: few hypotheses, an odd image, the plain L1 loss
        dict(name="track_7_odd", kind="track", sizes="317x239", focal=260.0, views=7, faces=40000, ssim=0.0),
        # serving: one render request against a dense resident map
        dict(name="render_1", kind="render", sizes="1200x680", focal=0.0, views=1, faces=2000000),
        # serving: a batch of render requests of the stream's three resolutions
        dict(name="render_9", kind="render", sizes="256x256,640x480,1200x680", focal=0.0, views=9, faces=2000000),
        # the tracking and mapping loss of a batch of full-size views
        dict(name="loss_20", kind="loss", sizes="1200x680", focal=0.0, views=20, ssim=0.2),
        # keyframe selection: coverage, visible sets and co-visibility of the window's views
        dict(name="keyframes_8", kind="keyframes", sizes="640x480", focal=0.0, views=8, faces=300000),
        # an extracted mesh (shared vertices) with the opacity and window variants switched on
        dict(name="mesh_3_odd", kind="mesh", sizes="333x251,640x480,511x333", focal=400.0, views=3, faces=100000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes spread over the logarithm of each kind's range, odd ones included."""
    kind = rng.choice(["frame", "step", "step", "step", "mapping", "track", "track", "render", "render", "loss",
                       "keyframes", "mesh"])
    n_sizes = 1 if kind in ("frame", "track") else rng.randint(1, 3)
    sizes = []
    for _ in range(n_sizes):
        w = _log_int(rng, 64, 1200)
        sizes.append((w, max(40, min(680, int(w * rng.uniform(0.55, 1.0))))))
    focal = float(int(rng.uniform(0.5, 0.9) * sum(w for w, _ in sizes) / n_sizes))
    views = {"frame": 1, "step": _log_int(rng, 1, 20), "mapping": _log_int(rng, 1, 8), "track": _log_int(rng, 1, 64),
             "render": _log_int(rng, 1, 9), "loss": _log_int(rng, 1, 20), "keyframes": rng.randint(2, 8),
             "mesh": rng.randint(1, 6)}[kind]
    views = max(views, n_sizes)
    top = {"frame": 4000, "step": 1000000, "mapping": 300000, "track": 150000, "render": 2000000, "loss": 1,
           "keyframes": 300000, "mesh": 200000}[kind]
    pixels = sum(w * h for w, h in sizes) / n_sizes
    # a cost that stays below the largest listed case: (view, face) records and contributions
    top = min(top, int(6e6 / views), int(4e7 / (12e-6 * views * focal * focal) + 1)) if kind != "loss" else 1
    case = dict(kind=kind, sizes=",".join("%dx%d" % s for s in sizes), focal=focal, views=views)
    if kind != "loss":
        case["faces"] = _log_int(rng, min(500, top), max(top, 1))
    if kind in ("track", "loss"):
        case["ssim"] = rng.choice([0.0, 0.2, 0.2]) if kind == "track" else 0.2
    if kind == "step":
        case["scene"] = "room" if rng.random() < 0.8 else "triangles"
        if case["scene"] == "triangles":
            case["faces"] = min(case["faces"], max(100, int(0.15 * pixels)))
        case["tile"] = rng.choice(["16x8", "16x8", "16x8", "16x16", "8x8"])
        case["stage"] = rng.choice([64, 64, 128])
        case["persistent"] = rng.random() < 0.15
    return case


def work(case):
    """Bytes: the map, the targets and the poses read once; images, losses and gradients written
    once.  Flops: 35 per blended (pixel, face) contribution forward and 90 backward, 394 per pixel
    and channel of the D-SSIM loss, the contributions from the map's density in the view."""
    cams = _cams(case)
    px = float(sum(c[4] * c[5] for c in cams))
    kind, M = case["kind"], case.get("faces", 0)
    if kind == "loss":
        return {"bytes": 48.0 * px, "flops": 3 * 394.0 * px}
    verts = (M / 2 if kind == "mesh" else 3.0 * M)
    contrib = sum(_density(case) * M * c[0] * c[0] for c in cams)
    map_b = 28.0 * verts + (12.0 * M + 4.0 * M if kind == "mesh" else 0.0)
    images = 20.0 * px
    if kind == "render":
        return {"bytes": map_b + images, "flops": 35.0 * contrib}
    if kind == "keyframes":
        return {"bytes": map_b + images + len(cams) * M * 8.125, "flops": 35.0 * contrib}
    grads = 0.0 if kind == "track" else 28.0 * verts + (4.0 * M if kind == "mesh" else 0.0)
    targets = 16.0 * px / (len(cams) if kind == "track" else 1)
    b, f = map_b + images + targets + grads, 125.0 * contrib
    if kind == "mapping":
        b += 24.0 * px
    if kind == "mapping" or case.get("ssim", 0.0) > 0:
        f += 3 * 394.0 * px
    return {"bytes": b, "flops": f}


def _density(case):
    """Contributions per face and squared focal length (counted on the scenes these follow)."""
    if case["kind"] == "mesh":
        return 4.0 / case["faces"]
    if case["kind"] == "frame" or case.get("scene") == "triangles":
        return 3.0e-4
    return 12e-6


# --------------------------------------------------------------------------------------- inputs
def _cams(case):
    """[V, 6]: fx, fy, cx, cy, W, H; the views take the case's sizes in runs of equal length."""
    sizes = [tuple(int(x) for x in s.split("x")) for s in case["sizes"].split(",")]
    V = case["views"]
    out = []
    for v in range(V):
        W, H = sizes[v * len(sizes) // V]
        f = case["focal"] or FOCAL["%dx%d" % (W, H)]
        out.append((f, f, W / 2.0, H / 2.0, W, H))
    return np.array(out, np.float64)


def _look_at(eye, target):
    f = target - eye
    f = f / np.linalg.norm(f)
    right = np.cross(f, np.array([0.0, 0.0, 1.0]))
    right /= np.linalg.norm(right)
    R = np.stack([right, np.cross(f, right), f])
    return np.concatenate([R.reshape(-1), -R @ eye])


def _trajectory(rng, n):
    """Poses on a circle of 1.5 m in the room, each looking across it at a jittered point."""
    out = []
    for i in range(n):
        th = 2 * np.pi * i / n + rng.uniform(-0.1, 0.1)
        eye = np.array([1.5 * np.cos(th), 1.5 * np.sin(th), 1.5])
        target = np.array([-2.4 * np.cos(th), -2.0 * np.sin(th), rng.uniform(0.6, 2.2)])
        target[:2] += rng.normal(0, 0.3, 2)
        out.append(_look_at(eye, target))
    return np.array(out)


def _perturbed(rng, pose, n, trans=0.05, deg=3.0):
    """n poses within +-trans metres and +-deg degrees of ``pose``."""
    R0, t0 = pose[:9].reshape(3, 3), pose[9:]
    out = []
    for _ in range(n):
        axis = rng.normal(size=3)
        axis /= np.linalg.norm(axis)
        a = np.deg2rad(rng.uniform(-deg, deg))
        K = np.array([[0, -axis[2], axis[1]], [axis[2], 0, -axis[0]], [-axis[1], axis[0], 0]])
        Rd = np.eye(3) + np.sin(a) * K + (1 - np.cos(a)) * (K @ K)
        out.append(np.concatenate([(Rd @ R0).reshape(-1), Rd @ t0 + rng.uniform(-trans, trans, 3)]))
    return np.array(out)


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=torch.float32)


def _flat_triangles(g, n, lo, hi):
    """n planar triangles with sides U[lo, hi] (10% triangle-inequality margin), centroid at 0,
    rotated at random in their plane: [n, 3, 2]."""
    got = torch.empty(0, 3, device=DEV)
    while got.shape[0] < n:
        s = _uniform(g, lo, hi, 2 * n + 64, 3)
        longest = s.max(1).values
        got = torch.cat([got, s[s.sum(1) - longest > 1.1 * longest]])
    a, b, c = got[:n].unbind(1)
    cos_a = ((b * b + c * c - a * a) / (2 * b * c)).clamp(-1, 1)
    P = torch.zeros(n, 3, 2, device=DEV)
    P[:, 1, 0] = c
    P[:, 2, 0] = b * cos_a
    P[:, 2, 1] = b * (1 - cos_a * cos_a).sqrt()
    P -= P.mean(1, keepdim=True)
    psi = _uniform(g, 0, 2 * math.pi, n)
    cp, sp = psi.cos(), psi.sin()
    return torch.stack([P[..., 0] * cp[:, None] - P[..., 1] * sp[:, None],
                        P[..., 0] * sp[:, None] + P[..., 1] * cp[:, None]], -1)


def _tangents(n):
    helper = torch.where(n[:, 2:3].abs() < 0.9, torch.tensor([[0.0, 0.0, 1.0]], device=DEV),
                         torch.tensor([[1.0, 0.0, 0.0]], device=DEV))
    t1 = F.normalize(torch.linalg.cross(n, helper), dim=1)
    return t1, torch.linalg.cross(n, t1)


def _room_surfaces(rng):
    """Rows (corner, edge 1, edge 2, normal, radius) of the walls, 40 random boxes and spheres; a
    sphere's corner is its centre and its radius is positive."""
    lo, hi = np.array([-3.0, -2.5, 0.0]), np.array([3.0, 2.5, 3.0])
    rows, areas = [], []

    def box(bmin, bmax, inward):
        ext = bmax - bmin
        for axis in range(3):
            a1, a2 = [k for k in range(3) if k != axis]
            for corner0, sgn in ((bmin, -1.0), (bmax, 1.0)):
                corner = bmin.copy()
                corner[axis] = corner0[axis]
                e1, e2, n = np.zeros(3), np.zeros(3), np.zeros(3)
                e1[a1], e2[a2], n[axis] = ext[a1], ext[a2], (-sgn if inward else sgn)
                rows.append(np.concatenate([corner, e1, e2, n, [0.0]]))
                areas.append(ext[a1] * ext[a2])

    box(lo, hi, True)
    for _ in range(40):
        if rng.random() < 0.5:
            size = rng.uniform(0.2, 1.0, 3)
            c = np.array([rng.uniform(-2.4, 2.4), rng.uniform(-1.9, 1.9), size[2] / 2])
            box(c - size / 2, c + size / 2, False)
        else:
            r = rng.uniform(0.1, 0.5)
            c = np.array([rng.uniform(lo[0] + r, hi[0] - r), rng.uniform(lo[1] + r, hi[1] - r), rng.uniform(r, 3.0 - r)])
            rows.append(np.concatenate([c, np.zeros(9), [r]]))
            areas.append(4 * np.pi * r * r)
    return np.array(rows), np.array(areas)


def _smooth_colours(rng, pts):
    """Four random plane waves per channel, in [0, 1]: [3, N]."""
    out = []
    for _ in range(3):
        w = torch.as_tensor(rng.normal(0.0, 2.5, (3, 4)), dtype=torch.float32, device=DEV)
        ph = torch.as_tensor(rng.uniform(0, 2 * np.pi, 4), dtype=torch.float32, device=DEV)
        out.append((0.5 + 0.125 * torch.sin(pts @ w + ph).sum(1)).clamp(0, 1))
    return torch.stack(out)


def _room(rng, g, n):
    rows, areas = _room_surfaces(rng)
    which = torch.multinomial(torch.as_tensor(areas, dtype=torch.float32, device=DEV), n, replacement=True, generator=g)
    q = torch.as_tensor(rows, dtype=torch.float32, device=DEV)[which]
    d = F.normalize(torch.randn(n, 3, generator=g, device=DEV), dim=1)
    sphere = q[:, 12:13] > 0
    centre = torch.where(sphere, q[:, :3] + q[:, 12:13] * d,
                         q[:, :3] + _uniform(g, 0, 1, n, 1) * q[:, 3:6] + _uniform(g, 0, 1, n, 1) * q[:, 6:9])
    nrm = torch.where(sphere, d, q[:, 9:12])
    t1, t2 = _tangents(nrm)
    ang, phi = _uniform(g, 0, math.radians(10.0), n, 1), _uniform(g, 0, 2 * math.pi, n, 1)
    nrm = ang.cos() * nrm + ang.sin() * (phi.cos() * t1 + phi.sin() * t2)
    t1, t2 = _tangents(nrm)
    flat = _flat_triangles(g, n, 0.01, 0.05)
    pts = (centre[:, None] + flat[..., 0:1] * t1[:, None] + flat[..., 1:2] * t2[:, None]).reshape(-1, 3)
    return pts, _smooth_colours(rng, pts), _uniform(g, 0.5, 1.0, 3 * n), None, None


def _triangles(rng, g, n, cam):
    """Random triangles in front of the camera at the identity pose, depth 0.5-4 m, sides 2-10 cm."""
    z = _uniform(g, 0.5, 4.0, n)
    u, v = _uniform(g, 0, cam[4], n), _uniform(g, 0, cam[5], n)
    centre = torch.stack([(u - cam[2]) * z / cam[0], (v - cam[3]) * z / cam[1], z], 1)
    nrm = F.normalize(torch.randn(n, 3, generator=g, device=DEV), dim=1)
    t1, t2 = _tangents(nrm)
    flat = _flat_triangles(g, n, 0.02, 0.10)
    pts = (centre[:, None] + flat[..., 0:1] * t1[:, None] + flat[..., 1:2] * t2[:, None]).reshape(-1, 3)
    return pts, torch.rand(3, 3 * n, generator=g, device=DEV), _uniform(g, 0.3, 1.0, 3 * n), None, None


def _mesh(rng, g, n):
    """A height field over 6 x 5 m on a jittered grid of about n indexed faces, below the cameras."""
    k = max(2, int(round(math.sqrt(n / 2.0))) + 1)
    gx, gy = torch.meshgrid(torch.arange(k, device=DEV), torch.arange(k, device=DEV), indexing="ij")
    jit = _uniform(g, -0.2, 0.2, 2, k, k)
    x, y = -3.0 + 6.0 * (gx + jit[0]) / (k - 1), -2.5 + 5.0 * (gy + jit[1]) / (k - 1)
    pts = torch.stack([x, y, 0.4 + 0.2 * torch.sin(1.7 * x) * torch.cos(1.3 * y)], -1).reshape(-1, 3)
    i = (gx[:-1, :-1] * k + gy[:-1, :-1]).reshape(-1)
    faces = torch.stack([torch.stack([i, i + k, i + 1], 1), torch.stack([i + 1, i + k, i + k + 1], 1)], 1)
    faces = faces.reshape(-1, 3).to(torch.int32).contiguous()
    return pts, _smooth_colours(rng, pts), _uniform(g, 0.5, 1.0, k * k), faces, _uniform(g, 0.5, 1.5, faces.shape[0])


def _images(rng, g, cams):
    """Packed camera images: smooth colour plus sensor noise in [0, 1]; smooth depth around 2.5 m
    with 1% noise and a tenth of the pixels without a reading."""
    C, D = [], []
    for c in cams:
        W, H = int(c[4]), int(c[5])
        yy, xx = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float32),
                                torch.arange(W, device=DEV, dtype=torch.float32), indexing="ij")
        p = rng.uniform(0, 1, (4, 4, 3))
        wave = lambda q: sum(torch.sin((0.02 + 0.3 * q[i, 0]) * xx + (0.02 + 0.3 * q[i, 1]) * yy  # noqa: E731
                                       + 6.28 * q[i, 2]) for i in range(4))
        img = torch.stack([0.5 + 0.2 * wave(p[ch]) for ch in range(3)])
        C.append((img + 0.02 * torch.randn(3, H, W, generator=g, device=DEV)).clamp(0, 1).reshape(-1))
        d = (2.5 + 0.3 * wave(p[3])) * (1 + 0.01 * torch.randn(H, W, generator=g, device=DEV))
        D.append((d * (torch.rand(H, W, generator=g, device=DEV) >= 0.1)).reshape(-1))
    return torch.cat(C).contiguous(), torch.cat(D).contiguous()


def _sensor_normals(g, cams):
    """Packed unit normals facing the camera, a tenth of the pixels without one."""
    out = []
    for c in cams:
        HW = int(c[4]) * int(c[5])
        n = F.normalize(torch.randn(3, HW, generator=g, device=DEV), dim=0)
        n[2] = -n[2].abs()
        out.append((n * (torch.rand(HW, generator=g, device=DEV) >= 0.1)).reshape(-1))
    return torch.cat(out).contiguous()


def _inputs(case, seed):
    """The tensors of a case: cams, poses [V, 12], map (pos [N, 3], col [3, N], opa, faces, sigma) and
    the target images its kind compares with."""
    rng = np.random.default_rng(seed)
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    cams, kind = _cams(case), case["kind"]
    d = {"cams": cams}
    if kind == "loss":
        d["tc"], d["td"] = _images(rng, g, cams)
        d["C"] = (d["tc"] + 0.05 * torch.randn(d["tc"].shape, generator=g, device=DEV)).clamp(0, 1)
        d["D"] = (2.5 + 0.5 * torch.randn(d["td"].shape, generator=g, device=DEV)).clamp_min(0.3)
        return d
    if kind == "frame" or case.get("scene") == "triangles":
        m = _triangles(rng, g, case["faces"], cams[0])
        poses = _perturbed(rng, np.array([1, 0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0.0]), len(cams), 0.02, 1.0)
    elif kind == "mesh":
        m = _mesh(rng, g, case["faces"])
        poses = _trajectory(rng, len(cams))
    else:
        m = _room(rng, g, case["faces"])
        poses = _trajectory(rng, len(cams))
        if kind == "track":
            poses = _perturbed(rng, poses[0], len(cams))
    d["pos"], d["col"], d["opa"], d["faces"], d["sigma"] = m
    d["poses"] = poses.astype(np.float32)
    if kind not in ("render", "keyframes"):
        d["tc"], d["td"] = _images(rng, g, cams[:1] if kind == "track" else cams)
    if kind == "mapping":
        d["tn"] = _sensor_normals(g, cams)
    return d


# -------------------------------------------------------------------------------------- the path
def _params(case):
    over = {}
    if "tile" in case:
        over["tile_w"], over["tile_h"] = (int(x) for x in case["tile"].split("x"))
        over["tris_per_stage"] = case["stage"]
        over["flags"] = ts.TS_FLAG_PERSISTENT if case["persistent"] else 0
    kind = case["kind"]
    if kind == "render":
        over["flags"] = ts.TS_FLAG_FORWARD_ONLY
    elif kind == "keyframes":
        over["flags"] = ts.TS_FLAG_STATS
    elif kind == "mesh":
        over["flags"] = ts.TS_FLAG_MIN_OPACITY | ts.TS_FLAG_FACE_SIGMA
    return ts.ts_default_params(**over)


def _capacity(case, cams):
    """(tile, face) pairs to make room for: the default holds 4 tiles per face of every view, which the
    large faces of random triangles and of coarse meshes exceed."""
    n = len(cams) * case["faces"]
    if case["kind"] == "mesh":
        return 4 * n + int(sum(c[4] * c[5] for c in cams))
    return 64 * n if case["kind"] == "frame" or case.get("scene") == "triangles" else 0


def _grad_map(m):
    """Gradient buffers of the map in one allocation, so that one fill clears them."""
    n = m.pos.shape[1]
    flat = torch.zeros(7 * n + (m.sigma.numel() if m.sigma is not None else 0), device=DEV)
    return flat, ts.Map(flat[:3 * n].view(3, n), flat[3 * n:6 * n].view(3, n), flat[6 * n:7 * n], m.faces,
                        flat[7 * n:] if m.sigma is not None else None)


def prepare(case, seed):
    d, p, kind = _inputs(case, seed), _params(case), case["kind"]
    s = {"kind": kind}
    if kind == "loss":
        r = ts.Rasterizer(d["cams"], 0, p)
        r.color.copy_(d["C"])
        r.depth.copy_(d["D"])
        return s | {"rast": r, "tc": d["tc"], "td": d["td"], "ssim": case["ssim"]}
    s["map"] = m = ts.Map(d["pos"].T.contiguous(), d["col"].contiguous(), d["opa"], d["faces"], d["sigma"])
    if kind == "track":
        W, H = int(d["cams"][0, 4]), int(d["cams"][0, 5])
        t = ts.Tracker(m, d["cams"][0], d["tc"].view(3, H, W), d["td"].view(H, W), d["poses"], p,
                       lambda_ssim=case["ssim"])
        t.capture()
        return s | {"tracker": t, "start": t.poses.clone()}
    s["poses"] = poses = ts.poses_tensor(d["poses"])
    if kind in ("render", "keyframes"):
        return s | {"rast": ts.Rasterizer(d["cams"], m.n_faces, p)}
    s["flat"], s["grad"] = _grad_map(m)
    s["tc"], s["td"] = d["tc"], d["td"]
    if kind in ("frame", "mesh"):
        return s | {"rast": ts.Rasterizer(d["cams"], m.n_faces, p, _capacity(case, d["cams"]))}
    extra = dict(lambda_ssim=0.2, tgt_normal=d["tn"], lambda_norm=0.05, lambda_equi=1.2) if kind == "mapping" else {}
    step = ts.MultiViewStep(m, d["cams"], poses, d["tc"], d["td"], p, s["grad"],
                            pair_capacity=_capacity(case, d["cams"]), **extra)
    step.capture()
    return s | {"step": step}


def run(s):
    kind = s["kind"]
    if kind == "loss":
        return list(s["rast"].pho_loss(s["tc"], s["td"], s["ssim"]))
    if kind == "track":
        t = s["tracker"]
        t.poses.copy_(s["start"])
        t.state.zero_()
        t.run(1)
        r = t.rast
        return [r.color, r.depth, r.alpha, t.loss(), r.dtau, t.poses]
    if kind == "render":
        return list(s["rast"].forward(s["map"], s["poses"]))
    if kind == "keyframes":
        r = s["rast"]
        out = list(r.forward(s["map"], s["poses"]))
        st = r.face_stats()
        return out + [st["area"], r.covisibility(st["visible"]), st["coverage"], st["visible"], st["n_visible"]]
    s["flat"].zero_()
    g = s["grad"]
    if kind in ("frame", "mesh"):
        r = s["rast"]
        r.forward(s["map"], s["poses"])
        loss, dC, dD = r.l1_loss(s["tc"], s["td"])
        r.backward(dC, dD, None, g)
        r.pose_grad()
        out = [r.color, r.depth, r.alpha, loss, r.dtau, g.pos, g.col, g.opa]
        return out + [g.sigma] if kind == "mesh" else out
    s["step"].run(1, use_graph=True)
    r = s["step"].rast
    out = [r.color, r.depth, r.alpha, r.loss_v, r.dtau, g.pos, g.col, g.opa]
    return out + [r.normal, r.nloss_v, s["step"].equi] if kind == "mapping" else out


# --------------------------------------------------------------------------- the same in 64 bits
MAX_ELEMENTS = 4.0e9   # (tile pixel, face) pairs one evaluation may take
CHUNK = 24_000_000
TW, TH = 16, 8


class _View:
    """One view in 64 bits: the visible faces' screen-space values as autograd functions of the map
    and the pose perturbation, and the depth-sorted face list of every tile."""

    def __init__(self, pos, col, opa, sigma, faces, cam, pose, tau, p, min_opacity, normals):
        R, t = pose[:9].reshape(3, 3), pose[9:]
        self.W, self.H = int(cam[4]), int(cam[5])
        with torch.no_grad():  # one float32 rounding per operation
            x, r = pos.float().T, pose.float()
            c32 = [((r[3 * i] * x[0] + r[3 * i + 1] * x[1]) + r[3 * i + 2] * x[2]) + r[9 + i] for i in range(3)]
            f, c = torch.as_tensor(cam[:2], device=DEV).float(), torch.as_tensor(cam[2:4], device=DEV).float()
            u32, v32 = f[0] * (c32[0] / c32[2]) + c[0], f[1] * (c32[1] / c32[2]) + c[1]
        vc = pos @ R.T + t
        vc = vc + tau[:3] + torch.linalg.cross(tau[3:].expand_as(vc), vc)  # left perturbation, first order
        oF = opa[faces].min(1).values if min_opacity else opa[faces].mean(1)
        with torch.no_grad():
            z, uu, vv = c32[2][faces], u32[faces], v32[faces]
            area2 = (uu[:, 1] - uu[:, 0]) * (vv[:, 2] - vv[:, 0]) - (uu[:, 2] - uu[:, 0]) * (vv[:, 1] - vv[:, 0])
            per = sum(((uu[:, (i + 1) % 3] - uu[:, i]) ** 2 + (vv[:, (i + 1) % 3] - vv[:, i]) ** 2).sqrt()
                      for i in range(3))
            x0, x1 = torch.ceil(uu.min(1).values - 0.5), torch.floor(uu.max(1).values - 0.5)
            y0, y1 = torch.ceil(vv.min(1).values - 0.5), torch.floor(vv.max(1).values - 0.5)
            vis = (z > p.z_near).all(1) & (area2.abs() / per >= p.r_min) & (oF >= p.alpha_min)
            vis &= (x0 <= x1) & (x1 >= 0) & (x0 <= self.W - 1) & (y0 <= y1) & (y1 >= 0) & (y0 <= self.H - 1)
            self.area = torch.where(vis, area2.abs().double() / 2, torch.zeros_like(oF))
            idx = torch.nonzero(vis).squeeze(1)
            key = ((z[:, 0] + z[:, 1]) + z[:, 2]) / 3
            idx = idx[torch.argsort(key[idx], stable=True)]  # depth order, ties by face
            self.idx = idx
            bx0, bx1 = x0[idx].clamp(min=0).long() // TW, x1[idx].clamp(max=self.W - 1).long() // TW
            by0, by1 = y0[idx].clamp(min=0).long() // TH, y1[idx].clamp(max=self.H - 1).long() // TH
            nx, ny = bx1 - bx0 + 1, by1 - by0 + 1
            n = nx * ny
            f = torch.repeat_interleave(torch.arange(len(idx), device=DEV), n)
            k = torch.arange(len(f), device=DEV) - torch.repeat_interleave(n.cumsum(0) - n, n)
            self.tx = (self.W + TW - 1) // TW
            tile = (by0[f] + k // nx[f]) * self.tx + bx0[f] + k % nx[f]
            tile, order = torch.sort(tile, stable=True)  # faces are in depth order: so is every tile's list
            self.list = f[order]
            n_tiles = self.tx * ((self.H + TH - 1) // TH)
            self.count = torch.bincount(tile, minlength=n_tiles)
            self.start = self.count.cumsum(0) - self.count
            self.by_count = torch.argsort(self.count, descending=True)
        fv = faces[idx]
        at = lambda value, q: value.double() + (q - q.detach())  # noqa: E731  (value with q's derivative)
        vis_vc = torch.stack([at(c32[k][fv], vc[:, k][fv]) for k in range(3)], 2)
        u = at(u32[fv], cam[0] * vis_vc[..., 0] / vis_vc[..., 2] + cam[2])
        v = at(v32[fv], cam[1] * vis_vc[..., 1] / vis_vc[..., 2] + cam[3])
        cols = [u, v, vis_vc[..., 2], col[:, fv].permute(1, 0, 2).reshape(len(idx), 9), oF[idx][:, None]]
        cols.append(sigma[idx][:, None] if sigma is not None else torch.full((len(idx), 1), p.sigma, device=DEV,
                                                                               dtype=torch.float64))
        if normals:
            nn = F.normalize(torch.linalg.cross(vis_vc[:, 1] - vis_vc[:, 0], vis_vc[:, 2] - vis_vc[:, 0]), dim=1)
            turned = (nn.detach() * vis_vc.detach().sum(1)).sum(1, keepdim=True) > 0
            cols.append(torch.where(turned, -nn, nn))
        self.screen = torch.cat(cols, 1)  # [visible, 17 (+ 3)]: u, v, z of the vertices, c, o_F, sigma, n
        self.p, self.normals = p, normals

    def chunks(self):
        """Tiles by falling list length, as many at a time as fit CHUNK (pixel, face) pairs."""
        counts = self.count[self.by_count].tolist()
        k = 0
        while k < len(counts) and counts[k] > 0:
            m = max(1, min(len(counts) - k, CHUNK // (counts[k] * TW * TH)))
            yield self.by_count[k:k + m], counts[k]
            k += m

    def elements(self):
        return float(self.count.sum()) * TW * TH

    def blend(self, S, tiles, L):
        """Composite ``tiles`` from the screen-space rows S: pixel offsets [T, 128], image values
        [channels, T, 128] (colour, depth, opacity and the normal), the pixels inside the image and
        the blended entries."""
        p = self.p
        i = torch.arange(L, device=DEV)
        have = i[None] < self.count[tiles][:, None]
        f = self.list[(self.start[tiles][:, None] + i[None]).clamp(max=max(len(self.list) - 1, 0))]
        r = S[f][..., None]  # [T, L, k, 1]
        q = torch.arange(TW * TH, device=DEV)
        px = (tiles % self.tx)[:, None] * TW + q[None] % TW
        py = (tiles // self.tx)[:, None] * TH + q[None] // TW
        X, Y = px[:, None].double() + 0.5, py[:, None].double() + 0.5
        u, v = [r[:, :, k] for k in range(3)], [r[:, :, 3 + k] for k in range(3)]
        D2 = (u[1] - u[0]) * (v[2] - v[0]) - (u[2] - u[0]) * (v[1] - v[0])
        ln = [torch.sqrt((u[(k + 1) % 3] - u[k]) ** 2 + (v[(k + 1) % 3] - v[k]) ** 2) for k in range(3)]
        per = ln[0] + ln[1] + ln[2]
        lam = [None] * 3
        m = None
        for k in range(3):
            j = (k + 1) % 3
            lam[(k + 2) % 3] = ((u[j] - u[k]) * (Y - v[k]) - (v[j] - v[k]) * (X - u[k])) / D2
            e = per / ln[k] * lam[(k + 2) % 3]
            m = e if m is None else torch.minimum(m, e)
        inside = (m > 0) & have[..., None]
        al = r[:, :, 18] * torch.where(inside, m, torch.ones_like(m)) ** r[:, :, 19]
        al = al.clamp(max=p.alpha_max)
        ok = inside & (al >= p.alpha_min)
        a = torch.where(ok, al, torch.zeros_like(al))
        logt = torch.log1p(-a.detach()).cumsum(1)
        ok = ok & ((ok & (torch.exp(logt) < p.T_min)).cumsum(1) == 0)
        a = a * ok
        lt = torch.log1p(-a)
        w = a * torch.exp(lt.cumsum(1) - lt)
        T = torch.exp(lt.sum(1))
        out = []
        for ch in range(3):
            c = lam[0] * r[:, :, 9 + 3 * ch] + lam[1] * r[:, :, 10 + 3 * ch] + lam[2] * r[:, :, 11 + 3 * ch]
            out.append((w * c).sum(1) + T * p.bg[ch])
        out.append((w * (lam[0] * r[:, :, 6] + lam[1] * r[:, :, 7] + lam[2] * r[:, :, 8])).sum(1))
        out.append(1 - T)
        if self.normals:
            out += [(w * r[:, :, 20 + k]).sum(1) for k in range(3)]
        return py * self.W + px, torch.stack(out), (px < self.W) & (py < self.H), (f, ok)

    def images(self, coverage=None):
        """The view's images [channels, H * W] (no gradient); counts blended pixels into coverage."""
        img = torch.zeros(8 if self.normals else 5, self.H * self.W, dtype=torch.float64, device=DEV)
        for ch in range(3):
            img[ch] = self.p.bg[ch]
        with torch.no_grad():
            S = self.screen.detach()
            for tiles, L in self.chunks():
                o, val, inimg, (f, ok) = self.blend(S, tiles, L)
                img[:, o[inimg]] = val[:, inimg]
                if coverage is not None:
                    coverage.index_add_(0, self.idx[f.reshape(-1)], (ok & inimg[:, None]).sum(2).reshape(-1))
        return img

    def backward(self, dimg):
        """Backpropagate the image gradients [channels, H * W] into the map and the perturbation."""
        S = self.screen.detach().requires_grad_()
        for tiles, L in self.chunks():
            o, val, inimg, _ = self.blend(S, tiles, L)
            g = dimg[:, torch.where(inimg, o, torch.zeros_like(o))] * inimg
            val.backward(g)
        self.screen.backward(S.grad if S.grad is not None else torch.zeros_like(S))


def _ssim_mean(x, y):
    """Mean SSIM of [3, H, W] images: 11 x 11 Gaussian window of sigma 1.5, zeros outside."""
    k = torch.exp(-torch.arange(-5, 6, dtype=torch.float64, device=DEV) ** 2 / (2 * 1.5 ** 2))
    k = k / k.sum()

    def blur(a):
        pad = F.pad(a, (5, 5, 0, 0))
        a = sum(k[i] * pad[..., i:i + a.shape[-1]] for i in range(11))
        pad = F.pad(a, (0, 0, 5, 5))
        return sum(k[i] * pad[..., i:i + a.shape[-2], :] for i in range(11))

    mx, my = blur(x), blur(y)
    sx, sy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    C1, C2 = 0.01 ** 2, 0.03 ** 2
    return ((2 * mx * my + C1) * (2 * sxy + C2) / ((mx * mx + my * my + C1) * (sx + sy + C2))).mean()


def _loss_gradients(img, tc, td, tn, ssim, W, H):
    """Loss and normal loss of one view's images [channels, HW] and the gradient of their mapping
    loss (lambda_dep 0.05, lambda_norm 0.05)."""
    x = img.detach().requires_grad_()
    HW = W * H
    c, t = x[:3], tc.view(3, HW)
    loss = (1 - ssim) * (c - t).abs().sum() / (3 * HW) + 0.05 * ((x[3] - td).abs() * (td > 0)).sum() / HW
    if ssim > 0:
        loss = loss + ssim * (1 - _ssim_mean(c.view(3, H, W), t.view(3, H, W)))
    total, nloss = loss, torch.zeros((), device=DEV, dtype=torch.float64)
    if tn is not None:
        n = tn.view(3, HW)
        nloss = ((1 - (x[5:8] * n).sum(0)) * (n != 0).any(0)).sum() / HW
        total = total + 0.05 * nloss
    total.backward()
    return loss.detach(), nloss.detach(), x.grad


def _exp_left(pose, step):
    """Exp(-step) o pose with step = (rho, theta)."""
    A = torch.zeros(4, 4, dtype=torch.float64)
    s = -step.cpu()
    A[:3, 3] = s[:3]
    A[0, 1], A[0, 2], A[1, 0], A[1, 2], A[2, 0], A[2, 1] = -s[5], s[4], s[5], -s[3], -s[4], s[3]
    T = torch.eye(4, dtype=torch.float64)
    T[:3, :3], T[:3, 3] = pose[:9].cpu().reshape(3, 3), pose[9:].cpu()
    Q = torch.linalg.matrix_exp(A) @ T
    return torch.cat([Q[:3, :3].reshape(-1), Q[:3, 3]])


def _equilateral(pos, faces):
    p = pos[faces]
    e = 0.0
    for n in range(3):
        a, b = p[:, (n + 1) % 3] - p[:, n], p[:, (n + 2) % 3] - p[:, n]
        e = e + ((a * b).sum(1) / (a.norm(dim=1) * b.norm(dim=1)) - 0.5) ** 2
    return (e / 3).mean()


def exact(case, seed):
    d, kind = _inputs(case, seed), case["kind"]
    cams = d["cams"]
    ssim = case.get("ssim", 0.2 if kind == "mapping" else 0.0)
    off = np.concatenate([[0], np.cumsum(cams[:, 4] * cams[:, 5])]).astype(int)
    if kind == "loss":
        C, D, tc, td = (d[k].double() for k in ("C", "D", "tc", "td"))
        loss, dC, dD = [], [], []
        for v, c in enumerate(cams):
            a, b = off[v], off[v + 1]
            img = torch.cat([C[3 * a:3 * b].view(3, -1), D[None, a:b]])
            lv, _, g = _loss_gradients(img, tc[3 * a:3 * b], td[a:b], None, ssim, int(c[4]), int(c[5]))
            loss.append(lv)
            dC.append(g[:3].reshape(-1))
            dD.append(g[3])
        return [torch.stack(loss), torch.cat(dC), torch.cat(dD)]
    p = _params(case)
    train = kind not in ("render", "keyframes")
    leaf = lambda t: t.double().detach().requires_grad_(train)  # noqa: E731
    pos, col, opa = leaf(d["pos"]), leaf(d["col"]), leaf(d["opa"])
    sigma = leaf(d["sigma"]) if d["sigma"] is not None else None
    M = d["faces"].shape[0] if d["faces"] is not None else d["pos"].shape[0] // 3
    faces = d["faces"].long() if d["faces"] is not None else torch.arange(3 * M, device=DEV).view(M, 3)
    poses = torch.as_tensor(d["poses"], device=DEV).double()
    tau = torch.zeros(len(cams), 6, dtype=torch.float64, device=DEV, requires_grad=train)
    normals = kind == "mapping"
    imgs, loss, nloss, areas, cover, elements = [], [], [], [], [], 0.0
    for v, c in enumerate(cams):
        view = _View(pos, col, opa, sigma, faces, c, poses[v], tau[v], p, kind == "mesh", normals)
        elements += view.elements() * (3.0 if train else 1.0)
        if elements / (v + 1) * len(cams) > MAX_ELEMENTS:
            return None
        cov = torch.zeros(M, dtype=torch.long, device=DEV) if kind == "keyframes" else None
        img = view.images(cov)
        imgs.append(img)
        areas.append(view.area)
        cover.append(cov)
        if not train:
            continue
        a, b = (0, off[1]) if kind == "track" else (off[v], off[v + 1])
        tn = d["tn"][3 * a:3 * b].double() if normals else None
        lv, nv, g = _loss_gradients(img, d["tc"][3 * a:3 * b].double(), d["td"][a:b].double(), tn, ssim, view.W, view.H)
        loss.append(lv)
        nloss.append(nv)
        view.backward(g)
        del view
    packed = [torch.cat([i[:3].reshape(-1) for i in imgs]), torch.cat([i[3] for i in imgs]),
              torch.cat([i[4] for i in imgs])]
    if kind == "render":
        return packed
    if kind == "keyframes":
        s = torch.stack([c > 0 for c in cover]).double()
        both = s @ s.T
        n = s.sum(1)
        either = n[:, None] + n[None] - both
        iou = torch.where(either > 0, both / either.clamp(min=1), torch.zeros_like(both))
        return packed + [torch.stack(areas), iou, None, None, None]
    if kind == "track":
        lr = torch.tensor([0.001] * 3 + [0.003] * 3, dtype=torch.float64, device=DEV)
        step = lr * tau.grad / (tau.grad.abs() + 1e-8)  # the first step of Adam
        moved = torch.stack([_exp_left(poses[v], step[v]) for v in range(len(cams))])
        return packed + [torch.stack(loss), tau.grad, moved]
    out = packed + [torch.stack(loss), tau.grad]
    equi = None
    if kind == "mapping":
        equi = _equilateral(pos, faces)
        (1.2 * equi).backward()
    out += [pos.grad.T.contiguous(), col.grad, opa.grad]
    if kind == "mesh":
        out.append(sigma.grad)
    if kind == "mapping":
        out += [torch.cat([i[5:8].reshape(-1) for i in imgs]), torch.stack(nloss), equi.detach().view(1)]
    return out
