"""The work that programs have this framework do, as cases to be measured.

A case is one pass of a program through the public entry points (``paper_2309_16818_gb300.mem``
and ``.inpaint``): a mapping node fuses the scans or images that arrived since the last
publication and reads the map out; an allocation-free loop fuses into its own layers; a batch of
simulated robots takes a few steps and reads every map; a plugin derives layers; crops are
inpainted, and the inpainting network is trained.

The sensors are simulated here on the GPU (rays cast against a procedural terrain, smooth random
images), from the case's seed alone. ``exact`` restates what a pass computes in 64 bits; the
decisions the library states as fixed float32 sequences (cell, gate, pixel, visibility) are taken
with the same float32 operations, because another decision would be another result.
"""
import math

import numpy as np
import torch

from paper_2309_16818_gb300 import inpaint
from paper_2309_16818_gb300 import mem as M

SIGMA0, SIGMA1, GATE, Z_NEAR = 0.01, 0.002, 2.0, 0.05


def listed():
    return [
        # A small robot's 20k-point scans from host memory (page-locked), height and colour:
        # the smallest calls, where launches and latency count.
        dict(name="scans 20k host", kind="scans", W=200, res=0.04, n=20_000, calls=5, host=True),
        # A 64-beam LiDAR in a real-time loop that may not allocate: height only, into its own layers.
        dict(name="noalloc 131k", kind="noalloc", W=400, res=0.05, beams=64, az=2048, calls=4),
        # The multi-modal pose: 128-beam LiDAR + depth camera, colour and 20 class probabilities
        # into four layers of a 500 x 500 map that moves with the robot.
        dict(name="poses 569k", kind="poses", W=500, res=0.04, beams=128, az=2048, depth=1.0, classes=20,
             topk=0, probs="f32", calls=3, cleanup=False),
        # The same kind of robot with a network that sends its top three classes, odometry that
        # drifts and obstacles that move: drift compensation, ray-cast clean-up, ageing variance.
        dict(name="poses 142k cleanup", kind="poses", W=500, res=0.04, beams=64, az=1024, depth=0.5, classes=20,
             topk=3, probs="f32", calls=3, cleanup=True),
        # Wide rows: 64 BF16 features and 20 classes per point of a depth camera (Gaussian features
        # in BF16, exponential averages in F16).
        dict(name="features 64 307k", kind="features", W=400, res=0.03, depth=1.0, feats=64, classes=20, calls=2),
        # Simulated robots: many small maps, one call a step, colour and 16 BF16 features; every
        # map is read when the episode ends.
        dict(name="batch 64 maps", kind="batch", maps=64, W=200, res=0.05, lo=5_000, hi=60_000, feats=16, calls=24),
        # Four cameras around the robot: 64 features and 20 classes per pixel into the cells they see.
        dict(name="cameras 4x848x480", kind="cameras", W=500, res=0.04, H=480, Wi=848, cams=4, feats=64, classes=20),
        # Post-processing of a published map: normals and the PCA layer of a 64-channel layer.
        dict(name="plugins 500", kind="plugins", W=500, res=0.04, feats=64, n_comp=3, dtype="f32"),
        # The diffusion fill of a training set's crops.
        dict(name="fill 256x256^2", kind="fill", B=256, H=256, Wc=256, tol=1e-6),
        # One map's odd-shaped regions inpainted as they come: fill, input preparation, network.
        dict(name="inpaint 6x200x136", kind="inpaint", B=6, H=200, Wc=136),
        # Inference over a batch of crops.
        dict(name="unet 256x256^2", kind="unet", B=256, H=256, Wc=256),
        # One training step.
        dict(name="train 16x256^2", kind="train", B=16, H=256, Wc=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(v):
    return int(v) // 2 * 2


def draw(rng):
    kind = rng.choice(["scans", "noalloc", "poses", "poses", "features", "batch", "cameras", "plugins", "fill",
                       "inpaint", "unet", "train"])
    W = _even(_log(rng, 150, 640))
    if kind == "scans":
        W = _even(_log(rng, 60, 400))
        return dict(kind=kind, W=W, res=round(8.0 / W, 4), n=_log(rng, 2_000, 60_000), calls=rng.randint(1, 6),
                    host=rng.random() < 0.5)
    if kind == "noalloc":
        return dict(kind=kind, W=W, res=round(20.0 / W, 4), beams=rng.choice([16, 32, 64, 128]),
                    az=rng.choice([512, 900, 1024, 1800, 2048]), calls=rng.randint(1, 4))
    if kind == "poses":
        return dict(kind=kind, W=W, res=round(rng.uniform(0.03, 0.08), 3), beams=rng.choice([16, 32, 64, 128]),
                    az=_log(rng, 500, 2048), depth=rng.choice([0.25, 0.5, 0.75, 1.0]), classes=rng.randint(4, 23),
                    topk=rng.choice([0, 0, 1, 3]), probs=rng.choice(["f32", "f32", "f16", "bf16"]),
                    calls=rng.randint(1, 3), cleanup=rng.random() < 0.4)
    if kind == "features":
        return dict(kind=kind, W=W, res=round(rng.uniform(0.02, 0.05), 3), depth=rng.choice([0.5, 0.75, 1.0]),
                    feats=rng.choice([32, 48, 64, 61]), classes=rng.randint(5, 20), calls=rng.randint(1, 2))
    if kind == "batch":
        W = _even(_log(rng, 64, 200))
        return dict(kind=kind, maps=_log(rng, 4, 64), W=W, res=round(10.0 / W, 4), lo=_log(rng, 500, 5_000),
                    hi=_log(rng, 10_000, 50_000), feats=rng.choice([8, 16, 16, 13]), calls=rng.randint(4, 24))
    if kind == "cameras":
        k = rng.uniform(0.3, 1.0)
        return dict(kind=kind, W=W, res=round(rng.uniform(0.03, 0.06), 3), H=int(480 * k), Wi=int(848 * k),
                    cams=rng.randint(1, 4), feats=rng.choice([16, 32, 64, 30]), classes=rng.randint(3, 20))
    if kind == "plugins":
        return dict(kind=kind, W=W, res=round(rng.uniform(0.03, 0.06), 3), feats=rng.choice([8, 16, 32, 33, 64]),
                    n_comp=rng.randint(1, 3), dtype=rng.choice(["f32", "bf16", "f16"]))
    if kind == "fill":
        return dict(kind=kind, B=_log(rng, 8, 200), H=rng.choice([64, 100, 128, 200, 256]),
                    Wc=rng.choice([64, 96, 130, 192, 256]), tol=rng.choice([1e-5, 1e-6]))
    B = {"inpaint": _log(rng, 1, 16), "unet": _log(rng, 2, 200), "train": _log(rng, 1, 16)}[kind]
    return dict(kind=kind, B=B, H=8 * rng.randint(8, 32), Wc=8 * rng.randint(8, 32))


# --------------------------------------------------------------------------- simulated sensors

def _gen(seed, *more):
    g = torch.Generator(device="cuda")
    s = int(seed) & 0x7FFFFFFF
    for m in more:
        s = (s * 1_000_003 + 7919 * int(m) + 12345) & 0x7FFFFFFF
    g.manual_seed(s)
    return g


def _rand(g, *shape, lo=0.0, hi=1.0, dtype=torch.float32):
    return torch.rand(shape, generator=g, device="cuda", dtype=dtype) * (hi - lo) + lo


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device="cuda")


def _host_rng(seed, *more):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, *[int(m) for m in more]])


def _terrain(phi, psi, x, y):
    """Rolling ground with 0.2 m steps, as the framework's own synthetic terrain."""
    base = 0.3 * torch.sin(0.7 * x) * torch.cos(0.5 * y)
    return base + 0.2 * (torch.sin(2 * math.pi * (x * math.cos(phi) + y * math.sin(phi)) / 2.5 + psi) > 0)


def _ground(phi, psi, x, y):
    return float(_terrain(phi, psi, torch.tensor(float(x), dtype=torch.float64),
                          torch.tensor(float(y), dtype=torch.float64)))


def _rot_z(a):
    c, s = math.cos(a), math.sin(a)
    return np.array([[c, -s, 0.0], [s, c, 0.0], [0.0, 0.0, 1.0]])


def _rot_y(a):
    c, s = math.cos(a), math.sin(a)
    return np.array([[c, 0.0, s], [0.0, 1.0, 0.0], [-s, 0.0, c]])


_OPTICAL = np.array([[0.0, 0.0, 1.0], [-1.0, 0.0, 0.0], [0.0, -1.0, 0.0]])


def _pose(R, t):
    T = np.eye(4)
    T[:3, :3] = R
    T[:3, 3] = t
    return T


def _hits(phi, psi, o, d, tmin, tmax, coarse):
    """Distance to the terrain along the unit rays d [N, 3] from o; NaN where there is none."""
    ts = [tmin * (tmax / tmin) ** (i / (coarse - 1)) for i in range(coarse)]
    hi = torch.full((d.shape[0],), float("nan"), device="cuda")
    lo = torch.full_like(hi, float("nan"))
    for i, t in enumerate(ts):
        below = o[2] + t * d[:, 2] <= _terrain(phi, psi, o[0] + t * d[:, 0], o[1] + t * d[:, 1])
        new = below & torch.isnan(hi)
        hi = torch.where(new, t, hi)
        lo = torch.where(new, ts[i - 1] if i else float("nan"), lo)
    for _ in range(12):
        mid = 0.5 * (lo + hi)
        under = o[2] + mid * d[:, 2] <= _terrain(phi, psi, o[0] + mid * d[:, 0], o[1] + mid * d[:, 1])
        hi, lo = torch.where(under, mid, hi), torch.where(under, lo, mid)
    return 0.5 * (lo + hi)


def _lidar_rays(beams, az, yaw):
    el = torch.deg2rad(torch.linspace(-25.0, 15.0, beams, device="cuda"))
    a = torch.arange(az, device="cuda") * (2 * math.pi / az) + yaw
    E, A = torch.meshgrid(el, a, indexing="ij")
    return torch.stack([E.cos() * A.cos(), E.cos() * A.sin(), E.sin()], -1).reshape(-1, 3)


def _camera_rays(w, h, f, R):
    v, u = torch.meshgrid(torch.arange(h, device="cuda") + 0.5, torch.arange(w, device="cuda") + 0.5, indexing="ij")
    d = torch.stack([(u - w / 2) / f, (v - h / 2) / f, torch.ones_like(u)], -1).reshape(-1, 3)
    d = d / d.norm(dim=1, keepdim=True)
    return d @ torch.tensor(R.T, dtype=torch.float32, device="cuda")


def _sensor_frame(T, p):
    R = torch.tensor(T[:3, :3], dtype=torch.float32, device="cuda")
    t = torch.tensor(T[:3, 3], dtype=torch.float32, device="cuda")
    return ((p - t) @ R).contiguous()


def _scan(seed, k, robot, phi, psi, beams, az, depth, lift=0.0):
    """One pose's cloud in the sensor's frame (LiDAR rays, then a depth camera's), misses as NaN,
    and the pose that odometry reports (`lift` metres off)."""
    g = _gen(seed, 11, k)
    x, y, yaw = robot
    base = np.array([x, y, _ground(phi, psi, x, y) + 0.6])
    T = _pose(_rot_z(yaw), base)
    parts = []
    if beams:
        d = _lidar_rays(beams, az, yaw)
        t = _hits(phi, psi, base, d, 0.5, 40.0, 64)
        parts.append((base, d, t))
    if depth:
        R = _rot_z(yaw) @ _rot_y(math.radians(30.0)) @ _OPTICAL
        cam = base + _rot_z(yaw) @ np.array([0.2, 0.0, -0.1])
        w, h = int(640 * depth), int(480 * depth)
        d = _camera_rays(w, h, 385.0 * depth, R)
        parts.append((cam, d, _hits(phi, psi, cam, d, 0.3, 6.0, 40)))
    pts = []
    for o, d, t in parts:
        r = t + _randn(g, t.shape[0]) * (0.01 + 0.002 * torch.nan_to_num(t))
        pts.append(torch.tensor(o, dtype=torch.float32, device="cuda") + r[:, None] * d)
    xyz = _sensor_frame(T, torch.cat(pts))
    T = T.copy()
    T[2, 3] += lift
    return xyz, T


def _path(seed, n, step=0.3):
    r = _host_rng(seed, 3)
    x, y, yaw, out = 0.0, 0.0, r.uniform(-math.pi, math.pi), []
    for _ in range(n):
        out.append((float(x), float(y), float(yaw)))
        yaw += math.radians(r.uniform(-15, 15))
        x, y = x + step * math.cos(yaw), y + step * math.sin(yaw)
    return out


def _world(seed):
    r = _host_rng(seed, 5)
    return float(r.uniform(0, 2 * math.pi)), float(r.uniform(0, 2 * math.pi))


def _colours(g, n):
    return torch.randint(0, 256, (n, 3), generator=g, device="cuda", dtype=torch.uint8)


_DT = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_CODE = {"f32": M.F32, "f16": M.F16, "bf16": M.BF16}


def _class_probs(g, n, k, dtype="f32"):
    return torch.softmax(3.0 * _randn(g, n, k), 1).to(_DT[dtype]).contiguous()


def _top(probs, k):
    p, i = torch.sort(probs, dim=1, descending=True, stable=True)
    out = torch.empty((probs.shape[0], 2 * k), device="cuda")
    out[:, 0::2], out[:, 1::2] = i[:, :k].float(), p[:, :k]
    return out


def _ground_points(seed, k, n, extent, phi, psi, xy=(0.0, 0.0)):
    """n noisy points, uniform over a square of the terrain, from a sensor 0.6 m above its centre."""
    g = _gen(seed, 13, k)
    r = _host_rng(seed, 17, k)
    s = np.array([xy[0], xy[1], _ground(phi, psi, *xy) + 0.6])
    p = _rand(g, n, 2, lo=-extent / 2, hi=extent / 2)
    px, py = p[:, 0] + xy[0], p[:, 1] + xy[1]
    v = torch.stack([px, py, _terrain(phi, psi, px, py)], 1) - torch.tensor(s, dtype=torch.float32, device="cuda")
    dist = v.norm(dim=1, keepdim=True)
    v = v + (v / dist) * _randn(g, n, 1) * (0.01 + 0.002 * dist)
    T = _pose(_rot_z(r.uniform(-math.pi, math.pi)), s)
    return _sensor_frame(T, v + torch.tensor(s, dtype=torch.float32, device="cuda")), T


def _smooth(g, c, h, w, sigma=8):
    """A smooth random field [h, w, c] of about unit variance."""
    n = _randn(g, 1, c, h // sigma + 3, w // sigma + 3)
    f = torch.nn.functional.interpolate(n, scale_factor=sigma, mode="bicubic", align_corners=False)
    return (1.4 * f[0, :, sigma:sigma + h, sigma:sigma + w]).permute(1, 2, 0).contiguous()


def _published(seed, W, res, phi, psi):
    """Height, variance and validity [W * W] of a map filled by earlier scans."""
    g = _gen(seed, 19)
    c = (torch.arange(W, device="cuda") - W // 2 + 0.5) * res
    Y, X = torch.meshgrid(c, c, indexing="ij")
    h = _terrain(phi, psi, X, Y) + 0.01 * _randn(g, W, W)
    s = _ground(phi, psi, 0.0, 0.0) + 0.6
    seen = torch.ones(W, W, dtype=torch.bool, device="cuda")
    for i in range(1, 48):  # cells the robot cannot see from where it stands were never filled
        t = i / 48.0
        seen &= s + t * (h - s) > _terrain(phi, psi, t * X, t * Y) - 0.02
    seen &= _rand(g, W, W) > 0.1
    var = _rand(g, W, W, lo=1e-5, hi=1e-3)
    return h.float().contiguous().view(-1), var.view(-1), seen.view(-1)


def _crops(seed, B, H, W, res=0.04):
    """Heights of B crops and the cells seen from a sensor above each (the rest is occluded)."""
    r = _host_rng(seed, 23)
    phi, psi = (torch.tensor(r.uniform(0, 2 * math.pi, (B, 1, 1)), dtype=torch.float32, device="cuda") for _ in "ab")

    def ground(x, y):
        s = torch.sin(2 * math.pi * (x * phi.cos() + y * phi.sin()) / 2.5 + psi)
        return 0.3 * torch.sin(0.7 * x) * torch.cos(0.5 * y) + 0.2 * (s > 0)

    x = ((torch.arange(W, device="cuda") - W / 2 + 0.5) * res).view(1, 1, W)
    y = ((torch.arange(H, device="cuda") - H / 2 + 0.5) * res).view(1, H, 1)
    z = ground(x, y)
    sx = torch.tensor(r.uniform(-0.25, 0.25, (B, 1, 1)) * W * res, dtype=torch.float32, device="cuda")
    sy = torch.tensor(r.uniform(-0.25, 0.25, (B, 1, 1)) * H * res, dtype=torch.float32, device="cuda")
    sz = ground(sx, sy) + torch.tensor(r.uniform(0.5, 1.2, (B, 1, 1)), dtype=torch.float32, device="cuda")
    seen = torch.ones_like(z, dtype=torch.bool)
    for i in range(1, 64):
        t = i / 64.0
        seen &= sz + t * (z - sz) > ground(sx + t * (x - sx), sy + t * (y - sy)) - 1e-4
    return z.contiguous(), seen.to(torch.uint8).contiguous()


_WIDTHS = (32, 64, 128, 128)


def _unet_shapes(cin=3, widths=_WIDTHS):
    a, b, c, d = widths
    convs = [(cin, a), (a, a), (a, b), (b, b), (b, c), (c, c), (c, d), (d, d), (d + c, c), (c, c), (c + b, b), (b, b),
             (b + a, a), (a, a)]
    out = []
    for i, o in convs:
        out += [(3, 3, i, o), (o,)]
    return out + [(a, 1), (1,)]


def _unet_params(seed):
    g = _gen(seed, 29)
    parts = []
    for s in _unet_shapes():
        if len(s) == 4:
            parts.append(_randn(g, *s).reshape(-1) * math.sqrt(2.0 / (9 * s[2])))
        elif len(s) == 2:
            parts.append(_randn(g, *s).reshape(-1) * (0.1 / math.sqrt(s[0])))
        else:
            parts.append(0.02 * _randn(g, *s))
    return torch.cat(parts)


def _unet_inputs(seed, B, H, W):
    """Inputs of the network as the preparation lays them out, with a rough fill of the holes."""
    z, known = _crops(seed, B, H, W)
    g = _gen(seed, 31)
    mean = z.mean(dim=(1, 2), keepdim=True)
    fill = torch.where(known > 0, z, z + 0.05 * _randn(g, B, H, W))
    hid = 1.0 - known.float()
    x3 = torch.stack([fill - mean, hid, known.float() * (0.1 * math.log(1e-4))], -1).contiguous()
    return x3, fill.contiguous(), z, (1 - known).contiguous()


# --------------------------------------------------------------------------- the cases' inputs

def _layer_specs(c):
    k = c["kind"]
    if k == "scans":
        return [dict(channels=3, rule=M.LATEST)]
    if k == "poses":
        K = c["classes"]
        return [dict(channels=3, rule=M.LATEST), dict(channels=K, rule=M.DIRICHLET, alpha0=1.0),
                dict(channels=K, rule=M.CLASSMAX), dict(channels=K, rule=M.EXPAVG, w=0.1)]
    if k == "features":
        return [dict(channels=3, rule=M.LATEST), dict(channels=c["feats"], rule=M.GAUSS, dtype=M.BF16),
                dict(channels=c["feats"], rule=M.EXPAVG, w=0.25, dtype=M.F16),
                dict(channels=c["classes"], rule=M.DIRICHLET, alpha0=1.0)]
    if k == "batch":
        return [dict(channels=3, rule=M.LATEST), dict(channels=c["feats"], rule=M.GAUSS, dtype=M.BF16)]
    if k == "cameras":
        return [dict(channels=c["feats"], rule=M.GAUSS), dict(channels=c["classes"], rule=M.DIRICHLET, alpha0=1.0),
                dict(channels=c["classes"], rule=M.CLASSMAX)]
    if k == "plugins":
        return [dict(channels=c["feats"], rule=M.LATEST, dtype=_CODE[c["dtype"]])]
    return []


def _map_options(c):
    if c["kind"] == "poses" and c["cleanup"]:
        return dict(time_var=1e-6, outlier_var=1e-5, drift_alpha=0.5, drift_min_points=100, ray_cleanup=True)
    return {}


def _cloud_calls(c, seed):
    """The point calls of a pass: (robot xy or None, xyz, pose, [(rows, layers)]) for each."""
    phi, psi = _world(seed)
    path = _path(seed, c["calls"])
    out = []
    for k in range(c["calls"]):
        g = _gen(seed, 37, k)
        if c["kind"] == "scans":
            xyz, T = _ground_points(seed, k, c["n"], c["W"] * c["res"], phi, psi, path[k][:2])
            src = [(_colours(g, c["n"]), [0])]
        elif c["kind"] == "poses":
            lift = float(_host_rng(seed, 41, k).uniform(-0.03, 0.03)) if c["cleanup"] else 0.0
            xyz, T = _scan(seed, k, path[k], phi, psi, c["beams"], c["az"], c["depth"], lift)
            n = xyz.shape[0]
            if c["topk"]:
                p = M.TopK(_top(_class_probs(g, n, c["classes"]), c["topk"]), c["classes"])
            else:
                p = _class_probs(g, n, c["classes"], c["probs"])
            src = [(_colours(g, n), [0]), (p, [1, 2, 3])]
        elif c["kind"] == "features":
            xyz, T = _scan(seed, k, path[k], phi, psi, 0, 0, c["depth"])
            n = xyz.shape[0]
            src = [(_colours(g, n), [0]), (_randn(g, n, c["feats"]).to(torch.bfloat16), [1, 2]),
                   (_class_probs(g, n, c["classes"]), [3])]
        else:  # noalloc
            xyz, T = _scan(seed, k, path[k], phi, psi, c["beams"], c["az"], 0)
            src = []
        out.append((path[k][:2], xyz, T, src))
    return out


def _batch_calls(c, seed):
    """The steps of a batch of simulated robots: (offsets, xyz, poses, sources) for each."""
    out = []
    r = _host_rng(seed, 43)
    worlds = [(float(a), float(b)) for a, b in r.uniform(0, 2 * math.pi, (c["maps"], 2))]
    phi = torch.tensor([w[0] for w in worlds], device="cuda", dtype=torch.float32)
    psi = torch.tensor([w[1] for w in worlds], device="cuda", dtype=torch.float32)
    for k in range(c["calls"]):
        n = np.floor(np.exp(r.uniform(math.log(c["lo"]), math.log(c["hi"]), c["maps"]))).astype(np.int64)
        off = np.concatenate([[0], np.cumsum(n)]).astype(np.int64)
        sxy, yaw = r.uniform(-1.0, 1.0, (c["maps"], 2)), r.uniform(-math.pi, math.pi, c["maps"])
        sz = [_ground(*worlds[b], *sxy[b]) + 0.6 for b in range(c["maps"])]
        T = np.stack([_pose(_rot_z(yaw[b]), [sxy[b, 0], sxy[b, 1], sz[b]]) for b in range(c["maps"])])
        g = _gen(seed, 47, k)
        N, ext = int(off[-1]), c["W"] * c["res"]
        b = torch.repeat_interleave(torch.arange(c["maps"], device="cuda"), torch.tensor(n, device="cuda"))
        s = torch.tensor(np.concatenate([sxy, np.array(sz)[:, None]], 1), dtype=torch.float32, device="cuda")[b]
        xy = s[:, :2] + _rand(g, N, 2, lo=-ext / 2, hi=ext / 2)
        step = torch.sin(2 * math.pi * (xy[:, 0] * phi[b].cos() + xy[:, 1] * phi[b].sin()) / 2.5 + psi[b]) > 0
        z = 0.3 * torch.sin(0.7 * xy[:, 0]) * torch.cos(0.5 * xy[:, 1]) + 0.2 * step
        v = torch.cat([xy, z[:, None]], 1) - s
        dist = v.norm(dim=1, keepdim=True)
        v = v + (v / dist) * _randn(g, N, 1) * (0.01 + 0.002 * dist)
        R = torch.tensor(T[:, :3, :3], dtype=torch.float32, device="cuda")[b]
        xyz = torch.einsum("ni,nij->nj", v, R).contiguous()
        out.append((off, xyz, T, [(_colours(g, N), [0]), (_randn(g, N, c["feats"]).to(torch.bfloat16), [1])]))
    return out


def _cameras(c, seed):
    phi, psi = _world(seed)
    z = _ground(phi, psi, 0.0, 0.0) + 0.6
    r = _host_rng(seed, 53)
    f = 420.0 * c["Wi"] / 848.0
    out = []
    for k in range(c["cams"]):
        a = k * math.pi / 2 + math.radians(r.uniform(-10, 10))
        R = _rot_z(a) @ _rot_y(math.radians(20.0 + r.uniform(-5, 5))) @ _OPTICAL
        g = _gen(seed, 59, k)
        out.append((_pose(R, [0.3 * math.cos(a), 0.3 * math.sin(a), z]), (f, f, c["Wi"] / 2.0, c["H"] / 2.0),
                    _smooth(g, c["feats"], c["H"], c["Wi"]),
                    torch.softmax(2.0 * _smooth(g, c["classes"], c["H"], c["Wi"]), 2).contiguous()))
    return out


def _features_layer(c, seed):
    """A feature layer with three strong directions, observed on most cells."""
    g = _gen(seed, 61)
    C, W2 = c["feats"], c["W"] ** 2
    q = torch.linalg.qr(_randn(g, C, C).double().cpu())[0].float().cuda()
    k = min(3, C)
    z = _randn(g, W2, k) * torch.tensor([3.0, 2.0, 1.0], device="cuda")[:k]
    f = torch.zeros(W2, C, device="cuda")
    for i in range(k):  # elementwise, so that the layer has the same bits on every run
        f += z[:, i:i + 1] * q[:, i]
    f = f + 0.05 * _randn(g, W2, C) + _randn(g, C)
    return f.to(_DT[c["dtype"]]).contiguous(), _rand(g, W2) < 0.7


_STREAM = []


def _stream():
    """The program's own stream, as every pass uses it (the library replays its kernel sequences
    from a graph on a stream that is not the default one)."""
    if not _STREAM:
        _STREAM.append(torch.cuda.Stream())
    return _STREAM[0]


def prepare(c, seed):
    k = c["kind"]
    s = {"case": c}
    layers = [M.Layer(**d) for d in _layer_specs(c)]
    if k in ("scans", "poses", "features"):
        s["calls"] = _cloud_calls(c, seed)
        if c.get("host"):
            s["calls"] = [(xy, x.cpu().pin_memory(), T, [(t.cpu().pin_memory(), l) for t, l in src])
                          for xy, x, T, src in s["calls"]]
        n = max(call[1].shape[0] for call in s["calls"])
        s["map"] = M.Map(c["W"], c["res"], layers, max_points=n + 1024, **_map_options(c))
    elif k == "noalloc":
        s["calls"] = _cloud_calls(c, seed)
        W2 = c["W"] ** 2
        s["layers"] = [torch.zeros(W2, device="cuda"), torch.zeros(W2, device="cuda")]
        s["layers"] += [torch.zeros(W2, dtype=torch.int32, device="cuda") for _ in range(3)]
    elif k == "batch":
        s["calls"] = _batch_calls(c, seed)
        n = max(call[1].shape[0] for call in s["calls"])
        s["map"] = M.Map(c["W"], c["res"], layers, n_maps=c["maps"], max_points=n + 1024)
    elif k in ("cameras", "plugins"):
        s["map"] = M.Map(c["W"], c["res"], layers, max_points=1024)
        h, var, seen = _published(seed, c["W"], c["res"], *_world(seed))  # a checkpoint, restored
        s["map"].set_layer(M.LAYER_HEIGHT, h)
        s["map"].set_layer(M.LAYER_VARIANCE, var)
        s["map"].set_layer(M.LAYER_VALID, seen.to(torch.uint8))
        if k == "cameras":
            s["cams"] = _cameras(c, seed)
        else:
            f, obs = _features_layer(c, seed)
            s["map"].set_layer(0, f)
            s["map"].set_layer(0, obs.to(torch.uint8), part=M.PART_OBSERVED)
    elif k in ("fill", "inpaint"):
        z, known = _crops(seed, c["B"], c["H"], c["Wc"])
        s["h"], s["known"] = torch.where(known > 0, z, 0.0).contiguous(), known
    if k in ("unet", "train"):
        s["x3"], s["fill"], s["target"], s["hidden"] = _unet_inputs(seed, c["B"], c["H"], c["Wc"])
        s["n_hidden"] = int(s["hidden"].sum().item())
    if k in ("inpaint", "unet", "train"):
        s["net"] = M.UNet()
        s["net"].set_params(_unet_params(seed))
    return s


# --------------------------------------------------------------------------- one pass

def _read_map(m, c, b=0):
    """Everything a fuse updates, as a consumer reads it."""
    out = {"height": m.get_layer(M.LAYER_HEIGHT, map_index=b), "var": m.get_layer(M.LAYER_VARIANCE, map_index=b),
           "valid": m.get_layer(M.LAYER_VALID, map_index=b), "n_acc": m.get_layer(M.LAYER_NACC, map_index=b),
           "n_rej": m.get_layer(M.LAYER_NREJ, map_index=b)}
    for i, d in enumerate(_layer_specs(c)):
        out["layer%d" % i] = m.get_layer(i, map_index=b)
        if d["rule"] == M.GAUSS:
            out["gvar%d" % i] = m.get_layer(i, M.PART_VAR, map_index=b)
    return out


def _read_batch(m, c):
    """The same of every map, each layer of all maps in one tensor."""
    n, W2 = c["maps"], c["W"] ** 2
    empty = lambda *shape, dtype=torch.float32: torch.empty(shape, dtype=dtype, device="cuda")  # noqa: E731
    out = {"height": empty(n, W2), "var": empty(n, W2), "valid": empty(n, W2, dtype=torch.uint8),
           "layer0": empty(n, W2, 3), "layer1": empty(n, W2, c["feats"], dtype=torch.bfloat16)}
    for b in range(n):
        m.get_layer(M.LAYER_HEIGHT, map_index=b, out=out["height"][b])
        m.get_layer(M.LAYER_VARIANCE, map_index=b, out=out["var"][b])
        m.get_layer(M.LAYER_VALID, map_index=b, out=out["valid"][b])
        m.get_layer(0, map_index=b, out=out["layer0"][b])
        m.get_layer(1, map_index=b, out=out["layer1"][b])
    return out


def run(s):
    c = s["case"]
    with torch.cuda.stream(_stream()):
        return _RUN[c["kind"]](s, c)


def _run_clouds(s, c):
    m = s["map"]
    fuse = m.fuse_pointcloud_host if c.get("host") else m.fuse_pointcloud
    for xy, xyz, T, src in s["calls"]:
        m.move(xy)
        fuse(xyz, T, src)
    return _read_map(m, c)


def _run_noalloc(s, c):
    for xy, xyz, T, _ in s["calls"]:
        M.fuse_pointcloud_noalloc(c["W"], c["res"], xyz, T, *s["layers"], time_var=1e-6)
    return dict(zip(("height", "var", "valid", "n_acc", "n_rej"), s["layers"]))


def _run_batch(s, c):
    for off, xyz, T, src in s["calls"]:
        s["map"].fuse_pointcloud_batch(off, xyz, T, src)
    return _read_batch(s["map"], c)


def _run_cameras(s, c):
    m, W2 = s["map"], c["W"] ** 2
    seen = []
    for T, K, feat, seg in s["cams"]:
        vis = torch.empty(W2, dtype=torch.uint8, device="cuda")
        pix = torch.empty(W2, dtype=torch.int32, device="cuda")
        m.fuse_image(c["H"], c["Wi"], K, T, [(feat, [0]), (seg, [1, 2])], vis=vis, pix=pix)
        seen += [vis, pix]
    return {"seen": seen, "layer0": m.get_layer(0), "gvar0": m.get_layer(0, M.PART_VAR),
            "observed": m.get_layer(0, M.PART_OBSERVED), "layer1": m.get_layer(1), "layer2": m.get_layer(2)}


def _run_plugins(s, c):
    normals, ok = s["map"].normals()
    proj, vals, vecs, mean = s["map"].pca(0, c["n_comp"])
    return {"normals": normals, "ok": ok, "proj": proj, "vals": vals, "vecs": vecs, "mean": mean}


def _run_fill(s, c):
    # the sweeps used are no result of the crop: they differ by a few from run to run
    return M.inpaint_diffusion(s["h"], s["known"], tol=c["tol"])[0]


def _run_inpaint(s, c):
    x3, fill, hidden, mean = inpaint.prepare(s["h"], s["known"])
    pred = s["net"].forward(x3, fill)
    return {"pred": pred, "fill": fill, "x3": x3, "hidden": hidden, "mean": mean}


def _run_unet(s, c):
    return s["net"].forward(s["x3"], s["fill"])


def _run_train(s, c):
    loss = s["net"].train_step(s["x3"], s["fill"], s["target"], s["hidden"], 1e-3, n_hidden=s["n_hidden"])
    return {"loss": loss, "params": s["net"].get_params()}


_RUN = {"scans": _run_clouds, "poses": _run_clouds, "features": _run_clouds, "noalloc": _run_noalloc,
        "batch": _run_batch, "cameras": _run_cameras, "plugins": _run_plugins, "fill": _run_fill,
        "inpaint": _run_inpaint, "unet": _run_unet, "train": _run_train}


# --------------------------------------------------------------------------- what a pass cannot do without

def _conv_flops(px):
    """Multiply-adds of the network's forward pass over px full-resolution cells, times two."""
    level = (0, 0, 1, 1, 2, 2, 3, 3, 2, 2, 1, 1, 0, 0)
    shapes = [s for s in _unet_shapes() if len(s) == 4]
    return sum(2.0 * 9 * s[2] * s[3] * px / 4 ** l for s, l in zip(shapes, level)) + 2.0 * _WIDTHS[0] * px


def work(c):
    """Bytes: the pass's inputs read once, and what it returns read from the map and written once."""
    k = c["kind"]
    if k in ("fill", "inpaint", "unet", "train"):
        px = float(c["B"] * c["H"] * c["Wc"])
        n_par = sum(math.prod(s) for s in _unet_shapes())
        if k == "fill":
            return {"bytes": px * (4 + 1 + 4), "flops": 0.0}
        if k == "inpaint":
            return {"bytes": px * (4 + 1 + 4 + 4 + 12 + 1) + 2 * n_par, "flops": _conv_flops(px)}
        if k == "unet":
            return {"bytes": px * (12 + 4 + 4) + 2 * n_par, "flops": _conv_flops(px)}
        return {"bytes": px * (12 + 4 + 4 + 1) + 4 * 7 * n_par, "flops": 3.0 * _conv_flops(px)}
    size = {M.F32: 4, M.BF16: 2, M.F16: 2}
    cell = 8 + 1 + 8  # height, variance, valid, counts, as they are returned
    for d in _layer_specs(c):
        S = 2 if d["rule"] == M.CLASSMAX else d["channels"]
        cell += S * size[d.get("dtype", M.F32)] + (4 if d["rule"] == M.GAUSS else 0)
    W2 = c["W"] ** 2
    if k == "cameras":
        # at most a cell's pixel of each image is read: about a tenth of the map is seen by one camera
        rows = 4 * (c["feats"] + c["classes"])
        return {"bytes": float(W2 * (8 + 2 * (cell - 17) + 1 + 5 * c["cams"]) + 0.1 * W2 * c["cams"] * rows),
                "flops": 0.0}
    if k == "plugins":
        row = c["feats"] * size[_CODE[c["dtype"]]]
        return {"bytes": float(W2 * (8 + 13 + row + 4 * c["n_comp"])),
                "flops": float(W2 * 0.7 * (c["feats"] ** 2 + 2 * c["feats"] * c["n_comp"]))}
    if k == "noalloc":
        return {"bytes": float(c["calls"] * c["beams"] * c["az"] * 12 + 2 * W2 * 20), "flops": 0.0}
    if k == "batch":
        n = c["maps"] * (c["hi"] - c["lo"]) / math.log(c["hi"] / c["lo"])
        return {"bytes": float(c["calls"] * n * (12 + 3 + 2 * c["feats"]) + 2 * c["maps"] * W2 * (cell - 12)),
                "flops": 0.0}
    if k == "scans":
        n, row = c["n"], 12 + 3
    else:
        cam = int(640 * c["depth"]) * int(480 * c["depth"])
        if k == "poses":
            n = c["beams"] * c["az"] + cam
            row = 12 + 3 + (8 * c["topk"] if c["topk"] else c["classes"] * (4 if c["probs"] == "f32" else 2))
        else:
            n, row = cam, 12 + 3 + 2 * c["feats"] + 4 * c["classes"]
    return {"bytes": float(c["calls"] * n * row + 2 * W2 * cell), "flops": 0.0}


# --------------------------------------------------------------------------- the same in 64 bits

def _r32(x):
    return x.float().double()


def _fma(a, b, c):
    return _r32(a * b + c)


def _f(x):
    """A host number as the float32 the library holds, in 64 bits."""
    return float(np.float32(x))


class _ExactMaps:
    """n maps of W x W cells in logical order, updated in 64 bits."""

    def __init__(self, c, n=1):
        self.W, self.res, self.n = c["W"], c["res"], n
        self.spec = _layer_specs(c)
        self.opt = _map_options(c)
        cells = n * self.W ** 2
        z = lambda *s: torch.zeros(s, dtype=torch.float64, device="cuda")  # noqa: E731
        self.h, self.v, self.acc, self.rej = z(cells), z(cells), z(cells), z(cells)
        self.valid = torch.zeros(cells, dtype=torch.bool, device="cuda")
        self.origin = np.zeros(2)
        self.L = []
        for d in self.spec:
            S = 2 if d["rule"] == M.CLASSMAX else d["channels"]
            self.L.append({"x": z(cells, S) + self._start(d, S), "gv": z(cells),
                           "obs": torch.zeros(cells, dtype=torch.bool, device="cuda")})

    @staticmethod
    def _start(d, S):
        if d["rule"] == M.DIRICHLET:
            return d["alpha0"]
        if d["rule"] == M.CLASSMAX:
            return torch.tensor([-1.0, 0.0], dtype=torch.float64, device="cuda")
        return 0.0

    def move(self, xy):
        s = [int(math.floor(abs(v) + 0.5) * (1 if v >= 0 else -1)) for v in (np.array(xy) - self.origin) / self.res]
        if s == [0, 0]:
            return
        W = self.W
        old = [torch.arange(W, device="cuda") + v for v in s]  # the cells that were here before
        inside = [(v >= 0) & (v < W) for v in old]
        keep = (inside[1][:, None] & inside[0][None, :]).view(-1)

        def shift(t, start):
            r = torch.roll(t.view(W, W, -1), (-s[1], -s[0]), (0, 1)).reshape(t.shape)
            return torch.where(keep.view(-1, *[1] * (t.dim() - 1)), r, torch.as_tensor(start, device="cuda").to(t.dtype))

        self.h, self.v, self.acc, self.rej = (shift(t, 0.0) for t in (self.h, self.v, self.acc, self.rej))
        self.valid = shift(self.valid, False)
        for d, L in zip(self.spec, self.L):
            L["x"] = shift(L["x"], self._start(d, L["x"].shape[1]))
            L["gv"], L["obs"] = shift(L["gv"], 0.0), shift(L["obs"], False)
        self.origin = self.origin + np.array(s) * self.res

    def fuse(self, xyz, T, src, index=None, range_min=0.1, range_max=50.0, time_var=None):
        W, half = self.W, self.W // 2
        T = np.asarray(T, dtype=np.float64).reshape(-1, 4, 4)
        R = torch.tensor(T[:, :3, :3].astype(np.float32), device="cuda").double()
        t = T[:, :3, 3].copy()
        t[:, :2] -= self.origin
        t = torch.tensor(t.astype(np.float32), device="cuda").double()
        b = torch.zeros(xyz.shape[0], dtype=torch.int64, device="cuda") if index is None else index
        fin = torch.isfinite(xyz).all(1)
        p = xyz.double()
        x, y, z = p[:, 0], p[:, 1], p[:, 2]
        rs = _r32(_fma(x, x, _fma(y, y, _r32(z * z))).sqrt())
        fin &= (rs >= _f(range_min)) & (rs <= _f(range_max))
        q = [_fma(R[b, i, 0], x, _fma(R[b, i, 1], y, _fma(R[b, i, 2], z, t[b, i]))) for i in range(3)]
        cx, cy = (torch.floor(_r32(v / _f(self.res))) for v in q[:2])
        keep = fin & (cx >= -half) & (cx < half) & (cy >= -half) & (cy < half)
        rows = keep.nonzero().view(-1)
        cell = b[rows] * W * W + (cy[rows].long() + half) * W + cx[rows].long() + half
        z, rs = q[2][rows], rs[rows]
        sm = _fma(torch.full_like(rs, _f(SIGMA1)), rs, _f(SIGMA0))
        vm = _r32(sm * sm)
        cells = self.h.shape[0]

        def total(v):
            return torch.zeros((cells, *v.shape[1:]), dtype=torch.float64, device="cuda").index_add_(0, cell, v)

        if self.opt.get("drift_alpha"):
            e = z - self.h[cell]
            ok = self.valid[cell] & ~(e * e > GATE ** 2 * (self.v[cell] + vm))
            if int(ok.sum()) >= self.opt["drift_min_points"]:
                self.h = torch.where(self.valid, self.h + _f(self.opt["drift_alpha"] * float(e[ok].mean())), self.h)
        d = z - self.h[cell]
        rej = self.valid[cell] & (d * d > GATE ** 2 * (self.v[cell] + vm))
        w = torch.where(rej, 0.0, 1.0 / vm)
        sw, swz, nr, n = total(w), total(w * z), total(rej.double()), total(torch.ones_like(z))
        na = n - nr
        P = sw + torch.where(self.valid, 1.0 / self.v, 0.0)
        new = na > 0
        self.h = torch.where(new, (swz + torch.where(self.valid, self.h / self.v, 0.0)) / P, self.h)
        self.v = torch.where(new, 1.0 / P, self.v)
        self.v = self.v + _f(self.opt.get("outlier_var", 0.0)) * nr
        self.valid = self.valid | new
        self.acc, self.rej = self.acc + na, self.rej + nr
        hit = n > 0
        N = n.clamp(min=1.0)
        for rowsrc, layers in src:
            if isinstance(rowsrc, M.TopK):
                ids, pr = rowsrc.pairs[:, 0::2].long(), rowsrc.pairs[:, 1::2].double()
                x = torch.zeros(ids.shape[0], rowsrc.K, dtype=torch.float64, device="cuda").scatter_add_(1, ids, pr)
            else:
                x = rowsrc
            x = x[rows].double()
            S = total(x)
            for l in layers:
                self._rule(self.spec[l], self.L[l], S, N, hit, x, cell)
        tv = self.opt.get("time_var", 0.0) if time_var is None else time_var
        self.v = torch.where(self.valid, self.v + _f(tv), self.v)

    @staticmethod
    def _rule(d, L, S, N, hit, x, cell):
        rule, obs, n = d["rule"], L["obs"], N[:, None]
        o = obs[:, None]
        if rule == M.LATEST:
            new = S / n
        elif rule == M.EXPAVG:
            w = _f(d["w"])
            new = torch.where(o, w * S / n + (1.0 - w) * L["x"], S / n)
        elif rule == M.GAUSS:
            s2, f2 = L["gv"][:, None], 1.0
            den = n * s2 + f2
            new = torch.where(o, (f2 * L["x"] + s2 * S) / den, S / n)
            gv = torch.where(obs, (f2 * s2 / den)[:, 0], f2 / N)
            L["gv"] = torch.where(hit, gv, L["gv"])
        elif rule == M.DIRICHLET:
            new = L["x"] + S
        else:
            top = x.max(1).values
            first = torch.where(x == top[:, None], torch.arange(x.shape[1], device="cuda"), 1 << 20).min(1).values
            best = torch.full_like(N, -math.inf).scatter_reduce(0, cell, top, "amax")
            at = torch.where(top == best[cell], first, 1 << 20).double()
            ids = torch.full_like(N, float(1 << 20)).scatter_reduce(0, cell, at, "amin")
            new = torch.stack([ids, best], 1)
        if d.get("dtype", M.F32) != M.F32:  # a stored value has its layer's type
            new = new.to(torch.bfloat16 if d["dtype"] == M.BF16 else torch.float16).double()
        L["x"] = torch.where(hit[:, None], new, L["x"])
        L["obs"] = obs | hit

    def out(self):
        z = torch.zeros_like(self.h)
        o = {"height": torch.where(self.valid, self.h, z), "var": torch.where(self.valid, self.v, z),
             "valid": self.valid.to(torch.uint8), "n_acc": self.acc.to(torch.int32), "n_rej": self.rej.to(torch.int32)}
        for i, (d, L) in enumerate(zip(self.spec, self.L)):
            o["layer%d" % i] = L["x"]
            if d["rule"] == M.GAUSS:
                o["gvar%d" % i] = L["gv"]
        return o


def _exact_cameras(c, seed):
    W, half, H, Wi = c["W"], c["W"] // 2, c["H"], c["Wi"]
    h, _, valid = _published(seed, W, c["res"], *_world(seed))
    h = h.double()
    res = _f(c["res"])
    iy, ix = (v.reshape(-1) for v in torch.meshgrid(torch.arange(W, device="cuda"), torch.arange(W, device="cuda"),
                                                   indexing="ij"))
    xc, yc = (_r32(((v - half).double() + 0.5) * res) for v in (ix, iy))
    F, K = c["feats"], c["classes"]
    mu, gv = torch.zeros(W * W, F, dtype=torch.float64, device="cuda"), torch.zeros(W * W, dtype=torch.float64,
                                                                                   device="cuda")
    obs = torch.zeros(W * W, dtype=torch.bool, device="cuda")
    alpha, cm = torch.ones(W * W, K, dtype=torch.float64, device="cuda"), torch.zeros(W * W, 2, dtype=torch.float64,
                                                                                     device="cuda")
    cm[:, 0] = -1.0
    seen = []
    for T, Kc, feat, seg in _cameras(c, seed):
        Rt = torch.tensor(T[:3, :3].T.astype(np.float32), device="cuda").double()
        tc = (-(T[:3, :3].T @ T[:3, 3])).astype(np.float32).astype(np.float64)
        X, Y, Z = (_fma(Rt[i, 0], xc, _fma(Rt[i, 1], yc, _fma(Rt[i, 2], h, torch.full_like(h, tc[i])))) for i in range(3))
        fx, fy, cx, cy = (_f(v) for v in Kc)
        u = torch.floor(_r32(_fma(torch.full_like(X, fx), _r32(X / Z), cx) + 0.5))
        v = torch.floor(_r32(_fma(torch.full_like(Y, fy), _r32(Y / Z), cy) + 0.5))
        cand = valid & (Z > _f(Z_NEAR)) & (u >= 0) & (u < Wi) & (v >= 0) & (v < H)
        e = cand.nonzero().view(-1)
        sx, sy = (int(min(max(math.floor(np.float32(T[i, 3]) / np.float32(c["res"])), -half), half - 1)) + half
                  for i in range(2))
        hc = _f(T[2, 3])
        ex, ey = ix[e], iy[e]
        dx, dy = ex - sx, ey - sy
        ax, ay = dx.abs(), dy.abs()
        major = torch.maximum(ax, ay)
        den = (dx * dx + dy * dy).double()
        dh = _r32(h[e] - hc)
        vis = torch.ones_like(e, dtype=torch.bool)
        x, y, err = torch.full_like(ex, sx), torch.full_like(ey, sy), ax - ay
        for k in range(1, int(major.max()) if e.numel() else 0):
            e2 = 2 * err
            mx, my = e2 >= -ay, e2 <= ax
            err = err - ay * mx + ax * my
            x, y = x + dx.sign() * mx, y + dy.sign() * my
            on = k < major
            q = (torch.where(on, y, 0) * W + torch.where(on, x, 0))
            tq = _r32(((x - sx) * dx + (y - sy) * dy).double() / den)
            vis &= ~(on & valid[q] & (h[q] >= _fma(tq, dh, hc)))
        e = e[vis]
        pix = v[e].long() * Wi + u[e].long()
        f, p = feat.view(-1, F)[pix].double(), seg.view(-1, K)[pix].double()
        s2, o = gv[e][:, None], obs[e][:, None]
        mu[e] = torch.where(o, (mu[e] + s2 * f) / (s2 + 1.0), f)
        gv[e] = torch.where(o, s2 / (s2 + 1.0), 1.0)[:, 0]
        alpha[e] += p
        best = p.max(1).values
        cm[e] = torch.stack([torch.where(p == best[:, None], torch.arange(K, device="cuda"), 1 << 20).min(1).values
                             .double(), best], 1)
        obs[e] = True
        one, pm = torch.zeros(W * W, dtype=torch.uint8, device="cuda"), torch.full((W * W,), -1, dtype=torch.int32,
                                                                                   device="cuda")
        one[e], pm[e] = 1, pix.to(torch.int32)
        seen += [one, pm]
    return {"seen": seen, "layer0": mu, "gvar0": gv, "observed": obs.to(torch.uint8), "layer1": alpha, "layer2": cm}


def _exact_plugins(c, seed):
    W = c["W"]
    h, _, valid = _published(seed, W, c["res"], *_world(seed))
    h, valid, res = h.double().view(W, W), valid.view(W, W), _f(c["res"])

    def slope(axis):
        def nb(d):
            on = torch.ones(W, W, dtype=torch.bool, device="cuda")
            on.select(axis, 0 if d < 0 else W - 1).fill_(False)
            return torch.roll(h, -d, axis), torch.roll(valid, -d, axis) & on
        (ha, va), (hb, vb) = nb(-1), nb(1)
        s = torch.where(va & vb, (hb - ha) / (2 * res), torch.where(vb, (hb - h) / res, (h - ha) / res))
        return s, va | vb

    (gx, okx), (gy, oky) = slope(1), slope(0)
    ok = (valid & okx & oky).view(-1)
    n = torch.stack([-gx, -gy, torch.ones_like(gx)], -1).view(-1, 3)
    n = torch.where(ok[:, None], n / n.norm(dim=1, keepdim=True), 0.0)
    f, obs = _features_layer(c, seed)
    x = f.double()[obs]
    mean = x.mean(0)
    vals, vecs = torch.linalg.eigh(((x - mean).T @ (x - mean) / x.shape[0]).cpu())
    vals, vecs = vals.flip(0)[:c["n_comp"]], vecs.flip(1)[:, :c["n_comp"]].T.contiguous()
    big = vecs.abs().argmax(1, keepdim=True)
    vecs = (vecs * vecs.gather(1, big).sign()).cuda()
    proj = torch.where(obs[:, None], (f.double() - mean) @ vecs.T, 0.0)
    return {"normals": n, "ok": ok.to(torch.uint8), "proj": proj, "vals": vals.cuda(), "vecs": vecs, "mean": mean}


def _exact_fill(h, known):
    """The harmonic fill by conjugate gradients from each crop's mean of known heights."""
    k = known.bool()
    h = h.double()
    n = k.sum((1, 2), keepdim=True)
    mean = torch.where(k, h, 0.0).sum((1, 2), keepdim=True) / n.clamp(min=1)
    u = torch.where(k, h, mean)
    deg = torch.full_like(h, 4.0)
    deg[:, 0] -= 1
    deg[:, -1] -= 1
    deg[:, :, 0] -= 1
    deg[:, :, -1] -= 1

    def lap(v):
        r = deg * v
        r[:, 1:] -= v[:, :-1]
        r[:, :-1] -= v[:, 1:]
        r[:, :, 1:] -= v[:, :, :-1]
        r[:, :, :-1] -= v[:, :, 1:]
        return r.masked_fill_(k, 0.0)

    dot = lambda a, b: (a * b).sum((1, 2), keepdim=True)  # noqa: E731
    r = -lap(u)
    p, rr = r.clone(), dot(r, r)
    for i in range(2500):
        q = lap(p)
        pq = dot(p, q)
        a = torch.where(pq > 0, rr / pq.clamp(min=1e-300), 0.0)
        u = u + a * p
        r = r - a * q
        new = dot(r, r)
        p = r + torch.where(rr > 0, new / rr.clamp(min=1e-300), 0.0) * p
        rr = new
        if i % 50 == 49 and float(rr.max()) < 1e-20:
            break
    return u


def _exact_net(params, x3, fill):
    F = torch.nn.functional
    p, o = [], 0
    for s in _unet_shapes():
        n = math.prod(s)
        p.append(params[o:o + n].view(s))
        o += n

    def conv(i, x):
        return F.relu(F.conv2d(x, p[2 * i].permute(3, 2, 0, 1), p[2 * i + 1], padding=1))

    def up(x, skip):
        return torch.cat([F.interpolate(x, scale_factor=2, mode="nearest"), skip], 1)

    x = x3.permute(0, 3, 1, 2)
    e1 = conv(1, conv(0, x))
    e2 = conv(3, conv(2, F.max_pool2d(e1, 2)))
    e3 = conv(5, conv(4, F.max_pool2d(e2, 2)))
    x = conv(7, conv(6, F.max_pool2d(e3, 2)))
    x = conv(9, conv(8, up(x, e3)))
    x = conv(11, conv(10, up(x, e2)))
    x = conv(13, conv(12, up(x, e1)))
    return fill + (x.permute(0, 2, 3, 1) @ p[28])[..., 0] + p[29]


def exact(c, seed):
    k = c["kind"]
    if k in ("scans", "poses", "features"):
        if k == "poses" and c["cleanup"]:
            return None  # which cells a ray clears is a decision of its own
        e = _ExactMaps(c)
        for xy, xyz, T, src in _cloud_calls(c, seed):
            e.move(xy)
            e.fuse(xyz, T, src)
        return e.out()
    if k == "noalloc":
        e = _ExactMaps(c)
        for _, xyz, T, _ in _cloud_calls(c, seed):
            e.fuse(xyz, T, [], time_var=1e-6)
        o = e.out()
        return {**o, "valid": o["valid"].to(torch.int32)}
    if k == "batch":
        n, W2 = c["maps"], c["W"] ** 2
        e = _ExactMaps(c, n)
        for off, xyz, T, src in _batch_calls(c, seed):
            count = torch.tensor(np.diff(off), device="cuda")
            e.fuse(xyz, T, src, torch.repeat_interleave(torch.arange(n, device="cuda"), count))
        o = e.out()
        return {"height": o["height"].view(n, W2), "var": o["var"].view(n, W2), "valid": o["valid"].view(n, W2),
                "layer0": o["layer0"].view(n, W2, -1), "layer1": o["layer1"].view(n, W2, -1)}
    if k == "cameras":
        return _exact_cameras(c, seed)
    if k == "plugins":
        return _exact_plugins(c, seed)
    px = c["B"] * c["H"] * c["Wc"]
    if k == "fill":
        if px > 2 << 20:  # many crops: minutes of 64-bit iterations
            return None
        z, known = _crops(seed, c["B"], c["H"], c["Wc"])
        return _exact_fill(torch.where(known > 0, z, 0.0), known)
    if px > 400_000:  # 64-bit convolutions of a large batch take too long
        return None
    params = _unet_params(seed).double()
    if k == "inpaint":
        z, known = _crops(seed, c["B"], c["H"], c["Wc"])
        kn = known.double()
        fill = _exact_fill(torch.where(known > 0, z, 0.0), known)
        mean = (z.double() * kn).sum((1, 2)) / kn.sum((1, 2)).clamp(min=1.0)
        x3 = torch.stack([fill - mean.view(-1, 1, 1), 1.0 - kn, kn * (0.1 * math.log(1e-4))], -1)
        return {"pred": _exact_net(params, x3, fill), "fill": fill, "x3": x3, "hidden": None, "mean": mean}
    x3, fill, target, hidden = _unet_inputs(seed, c["B"], c["H"], c["Wc"])
    if k == "unet":
        return _exact_net(params, x3.double(), fill.double())
    params.requires_grad_(True)
    d = (_exact_net(params, x3.double(), fill.double()) - target.double()) * hidden.double()
    loss = d.square().sum() / max(1, int(hidden.sum()))
    g, = torch.autograd.grad(loss, params)
    # the first step of Adam: both moments, corrected, are the gradient itself
    return {"loss": loss.detach().view(1), "params": params.detach() - 1e-3 * g / (g.abs() + 1e-8)}
