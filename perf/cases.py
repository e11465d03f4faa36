"""The work that users of this framework have it do, as cases that can be timed.

Each case is one pass through the public binding (``paper_1909_04631_gb300``) on inputs made from a seed:

- ``train``   the training set of one small scan through the allocation-free entry point;
- ``update``  one synchronous scan update of a map, then the read-off of the window of voxels around the sensor
              (mean and variance of the Dirichlet posterior), as a planner takes it; the ``form`` is the update's: hard
              labels, soft labels, the counting sensor model, per-class length scales, or the extended-block
              association;
- ``stream``  consecutive scans through the asynchronous entry point, one wait at the end, then the window;
- ``batch``   one batched update of independent maps with scans of mixed sizes, then each map's window;
- ``grad``    one training set into a map, held-out log-likelihood, and the gradient for l, sigma0 and every point;
- ``points``  Eq. (alpha_kernel) at arbitrary points of space, from a training set;
- ``readoff`` every read-off quantity at world points of a map restored from a snapshot.

Scenes are ray cast here on the GPU against boxes and a ground plane: a walled region, a street seen by a spinning
LiDAR, a furnished room seen by a depth camera.  Parameters are those of the paper's workloads (0.1 m voxels and
l = 0.3 m outdoors with 10 or 19 classes, 0.05 m and 0.15 m indoors with 11).
"""
import math

import numpy as np
import torch

import paper_1909_04631_gb300 as sb

DEV = "cuda"
SCENES = {
    # class count, voxel edge, free-sample spacing, sigma0, range limits
    "region": dict(classes=10, res=0.1, free_step=0.3, sigma0=1.0, min_range=0.0, max_range=100.0),
    "street": dict(classes=19, res=0.1, free_step=0.3, sigma0=0.1, min_range=0.0, max_range=50.0),
    "room": dict(classes=11, res=0.05, free_step=0.15, sigma0=0.1, min_range=0.3, max_range=8.0),
}
ALPHA0 = 0.001
# per-class length scales of the "scales" form: small classes get a tighter kernel, large flat ones a wider one
L_SCALES = (1.0, 1.0, 1.0, 1.15, 1.15, 1.0, 0.8, 0.8, 0.6, 0.6, 0.6, 1.0)


def listed():
    return [
        # a 2D or sparse sensor's sweep in a loop that may not allocate: latency and launches are all that counts
        dict(name="train_small", kind="train", scene="region", rays=1800, lr=3.0),
        # the paper's single ray-cast scan of a small walled region
        dict(name="region_scan", kind="update", scene="region", rays=10000, form="hard", lr=3.0, edge=8, host=False,
             side=100, height=24),
        # one 64-beam LiDAR revolution, synchronous: a robot that needs the map before its next decision
        dict(name="street_scan", kind="update", scene="street", rays=131072, form="hard", lr=3.0, edge=8, host=False,
             side=160, height=32),
        # the same sensor streamed along the street: throughput of the asynchronous path
        dict(name="street_stream", kind="stream", scene="street", rays=131072, scans=8, lr=3.0, side=160, height=32),
        # a 640x480 depth frame arriving in pinned host memory, indoors, fine voxels
        dict(name="room_frame", kind="update", scene="room", rays=307200, form="hard", lr=3.0, edge=8, host=True,
             side=120, height=40),
        # a server that keeps one map per robot: 16 scans of mixed sizes in one call
        dict(name="batch_mixed", kind="batch", scene="street", maps=16, n_min=5000, n_max=250000, lr=3.0,
             side=64, height=24),
        # the segmentation network's softmax instead of its most probable class
        dict(name="street_soft", kind="update", scene="street", rays=131072, form="soft", lr=3.0, edge=8, host=False,
             side=160, height=32),
        # the counting sensor model (the paper's S-CSM baseline map)
        dict(name="street_count", kind="update", scene="street", rays=131072, form="count", lr=3.0, edge=8, host=False,
             side=160, height=32),
        # class-dependent length scales
        dict(name="street_scales", kind="update", scene="street", rays=131072, form="scales", lr=3.0, edge=8,
             host=False, side=160, height=32),
        # one step of learning the kernel's parameters: training set in, held-out likelihood, gradients
        dict(name="region_grad", kind="grad", scene="region", points=2000000, scans=4, lr=3.0),
        # the continuous model queried off the voxel grid, a surface's worth of points
        dict(name="points_query", kind="points", scene="street", rays=131072, queries=200000, lr=3.0),
        # a planner reading a whole window of a restored map
        dict(name="window_readoff", kind="readoff", classes=19, extent=160, height=48, order="raster"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "update", "update", "update", "update", "stream", "batch", "grad", "points",
                       "readoff"])
    scene = rng.choice(["region", "street", "street", "room"])
    lr = rng.choice([3.0, 3.0, 3.0, 2.0, 2.5])
    if kind == "train":
        return dict(kind=kind, scene=rng.choice(["region", "room"]), rays=_log_int(rng, 200, 4000), lr=lr)
    if kind == "update":
        form = rng.choice(["hard", "hard", "soft", "count", "scales", "face"])
        edge = rng.choice([8, 8, 8, 4]) if form == "hard" else 8
        if form == "hard" and edge == 8:
            lr = rng.choice([lr, 4.0])  # a kernel wider than the paper's
        return dict(kind=kind, scene=scene, rays=_log_int(rng, 1500, 131072 if lr <= 3.0 else 40000), form=form, lr=lr,
                    edge=edge, host=rng.random() < 0.25, side=rng.randint(20, 160), height=rng.randint(8, 32))
    if kind == "stream":
        return dict(kind=kind, scene=scene, rays=_log_int(rng, 4000, 131072), scans=rng.randint(2, 8), lr=lr,
                    side=rng.randint(20, 160), height=rng.randint(8, 32))
    if kind == "batch":
        return dict(kind=kind, scene="street", maps=rng.randint(2, 16), n_min=2000, n_max=_log_int(rng, 8000, 250000),
                    lr=lr, side=rng.randint(20, 64), height=rng.randint(8, 24))
    if kind == "grad":
        return dict(kind=kind, scene=rng.choice(["region", "room"]), points=_log_int(rng, 3000, 2000000),
                    scans=rng.randint(1, 4), lr=lr)
    if kind == "points":
        return dict(kind=kind, scene=scene, rays=_log_int(rng, 3000, 131072), queries=_log_int(rng, 300, 200000),
                    lr=lr)
    return dict(kind=kind, classes=rng.randint(2, 24), extent=rng.randint(20, 160), height=rng.randint(8, 48),
                order=rng.choice(["raster", "cloud"]))


# ---------------------------------------------------------------- scenes and sensors
def _boxes(scene, rng):
    """(lo, hi, class) rows of a scene's solids; class 1 is the ground."""
    b = []

    def add(lo, hi, c):
        b.append(list(lo) + list(hi) + [c])

    if scene == "region":
        for lo, hi in (((-10.2, -10, 0), (-10, 10, 4)), ((10, -10, 0), (10.2, 10, 4)), ((-10, -10.2, 0), (10, -10, 4)),
                       ((-10, 10, 0), (10, 10.2, 4))):
            add(lo, hi, 2)
        for k in range(10):
            s = rng.uniform(0.4, 2.5, 3)
            a, r = rng.uniform(0, 2 * math.pi), rng.uniform(4.5, 8.0)
            c = (r * math.cos(a), r * math.sin(a))
            add((c[0] - s[0] / 2, c[1] - s[1] / 2, 0), (c[0] + s[0] / 2, c[1] + s[1] / 2, s[2]), 3 + k % 8)
    elif scene == "street":
        for side in (-1.0, 1.0):
            def strip(x0, x1, y0, y1, z0, z1, c):
                ya, yb = sorted((side * y0, side * y1))
                add((x0, ya, z0), (x1, yb, z1), c)

            x = -60.0
            while x < 75.0:  # facades, a fence or a low wall in the gaps
                seg, y0 = rng.uniform(8, 30), 8 + rng.uniform(0, 4)
                strip(x, x + seg, y0, y0 + 10, 0, rng.uniform(5, 20), 5)
                x += seg
                gap = rng.uniform(1, 6)
                strip(x, x + gap, 8.3, 8.5, 0, rng.uniform(0.6, 1.8), 6 if rng.random() < 0.5 else 19)
                x += gap
            x = -58.0 + rng.uniform(0, 8)
            while x < 75.0:  # trees, poles with signs
                y, th, rr = rng.uniform(6, 7), rng.uniform(2, 3), rng.uniform(1.0, 2.0)
                strip(x - 0.2, x + 0.2, y - 0.2, y + 0.2, 0, th, 8)
                strip(x - rr, x + rr, y - rr, y + rr, th, th + 1.6 * rr, 7)
                p = x + rng.uniform(3, 6)
                strip(p - 0.1, p + 0.1, 7.3, 7.5, 0, 6, 9)
                strip(p - 0.04, p + 0.04, 7.0, 7.8, 5, 5.8, 10)
                x += rng.uniform(8, 18)
            x = -60.0 + rng.uniform(0, 5)
            while x < 75.0:  # parked vehicles, people and two-wheelers on the pavement
                k = rng.random()
                ln, w, h, c = ((4.4, 1.8, 1.5, 11) if k < 0.7 else
                               (7.5, 2.4, 3.0, 12) if k < 0.85 else (5.0, 1.9, 2.1, 15))
                strip(x, x + ln, 3.7, 3.7 + w, 0.15, h, c)
                q = x + rng.uniform(0, 4)
                strip(q, q + 0.5, 5.4, 5.9, 0, 1.75, 16)
                strip(q + 2, q + 3.7, 5.3, 5.8, 0, 1.1, int(rng.choice([13, 14, 17])))
                x += ln + rng.uniform(0.5, 8)
    else:
        for lo, hi, c in (((-5, -4, 3), (5, 4, 3.2), 2), ((-5.2, -4, 0), (-5, 4, 3), 3), ((5, -4, 0), (5.2, 4, 3), 3),
                          ((-5, -4.2, 0), (5, -4, 3), 4), ((-5, 4, 0), (5, 4.2, 3), 4)):
            add(lo, hi, c)
        for k in range(18):  # furniture away from the camera's stand
            s = rng.uniform(0.3, 1.4, 3)
            a, r = rng.uniform(0, 2 * math.pi), rng.uniform(2.2, 3.6)
            c = (1.15 * r * math.cos(a), r * math.sin(a))
            add((c[0] - s[0] / 2, c[1] - s[1] / 2, 0), (c[0] + s[0] / 2, c[1] + s[1] / 2, s[2]), 5 + k % 7)
    return np.asarray(b, np.float64)


def _directions(scene, rays, rng):
    """Sensor-frame unit directions: a spinning LiDAR's rings, random rays of a region scan, or a pinhole image."""
    if scene == "room":
        h = max(2, int(round(math.sqrt(rays * 0.75))))
        w = max(2, rays // h)
        v, u = torch.meshgrid(torch.arange(h, device=DEV, dtype=torch.float64),
                              torch.arange(w, device=DEV, dtype=torch.float64), indexing="ij")
        d = torch.stack([torch.ones_like(u), -(u - (w - 1) / 2) / (0.82 * w), -(v - (h - 1) / 2) / (1.094 * h)], -1)
        return (d / d.norm(dim=-1, keepdim=True)).reshape(-1, 3)
    beams = max(4, min(128, int(round(math.sqrt(rays / 32.0)))))
    n_az = max(4, rays // beams)
    lo, hi = (-24.8, 2.0) if scene == "street" else (-15.0, 15.0)
    el = torch.linspace(math.radians(hi), math.radians(lo), beams, device=DEV, dtype=torch.float64)
    az = torch.arange(n_az, device=DEV, dtype=torch.float64) * (2 * math.pi / n_az) + rng.uniform(0, 0.01)
    e, a = torch.meshgrid(el, az, indexing="ij")
    return torch.stack([e.cos() * a.cos(), e.cos() * a.sin(), e.sin()], -1).reshape(-1, 3)


def _pose(scene, rng, at):
    yaw = rng.uniform(-math.pi, math.pi) if scene == "room" else math.radians(rng.normal(0, 1.0))
    T = np.eye(4)
    T[:2, :2] = [[math.cos(yaw), -math.sin(yaw)], [math.sin(yaw), math.cos(yaw)]]
    T[:3, 3] = {"street": (at + rng.uniform(0, 0.5), -1.75, 1.73), "region": (rng.uniform(-1, 1) + at, 0.3, 1.5),
                "room": (rng.uniform(-0.6, 0.6), rng.uniform(-0.6, 0.6), 1.4)}[scene]
    return T


def _ground_class(scene, y):
    if scene != "street":
        return torch.ones_like(y, dtype=torch.int32)
    a = y.abs()
    return torch.where(a < 3.5, 1, torch.where(a < 5.0, 2, torch.where(a < 8.0, 3, 4))).to(torch.int32)


def _scans(scene, rays, count, seed, keep=None):
    """`count` consecutive labelled scans of one scene: (points [n,3] f32, labels [n] i32, pose), on the GPU."""
    prm = SCENES[scene]
    rng = np.random.default_rng([seed, 11])
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    boxes = torch.from_numpy(_boxes(scene, rng)).to(DEV)
    out = []
    for i in range(count):
        T = _pose(scene, rng, float(i) if scene == "street" else 0.5 * i)
        ds = _directions(scene, rays if keep is None else 4 * keep[i] // 3 + 64, rng)
        Tt = torch.from_numpy(T).to(DEV)
        d, o = ds @ Tt[:3, :3].T, Tt[:3, 3]
        t = torch.where(d[:, 2] < -1e-9, -o[2] / d[:, 2], math.inf)
        cls = _ground_class(scene, o[1] + t.clamp(max=1e4) * d[:, 1])
        inv = 1.0 / torch.where(d.abs() < 1e-12, 1e-12, d)
        for b in boxes:
            t0, t1 = (b[:3] - o) * inv, (b[3:6] - o) * inv
            near, far = torch.minimum(t0, t1).amax(1), torch.maximum(t0, t1).amin(1)
            hit = (near > 0.05) & (near < far) & (near < t)
            t = torch.where(hit, near, t)
            cls = torch.where(hit, b[6].to(torch.int32), cls)
        ok = t < prm["max_range"]
        t, ds, cls = t[ok], ds[ok], cls[ok]
        t = t + 0.02 * torch.randn(t.shape, generator=gen, device=DEV, dtype=torch.float64)
        noise = torch.rand(t.shape, generator=gen, device=DEV) < 0.08
        other = torch.randint(1, prm["classes"] + 1, t.shape, generator=gen, device=DEV, dtype=torch.int32)
        lab = torch.where(noise, other, cls.clamp(1, prm["classes"])).contiguous()
        pts = (ds * t[:, None]).float()
        if keep is not None:  # a sensor of another resolution: some of the rays
            sel = torch.randperm(len(pts), generator=gen, device=DEV)[:keep[i]].sort().values
            pts, lab = pts[sel], lab[sel]
        out.append((pts.contiguous(), lab, T))
    return out


def _batch_sizes(case, seed):
    n = np.geomspace(case["n_min"], case["n_max"], case["maps"]).astype(int)
    return [int(v) for v in np.random.default_rng([seed, 5]).permutation(n)]


# ---------------------------------------------------------------- plain reference of the definition (64 bits)
def _training(scene, pts, lab, T, probs=None):
    """Steps a1-a3 of one scan: (xyz f32 [P,3], class [P], weights f64 [P,K+1] or None),
    ordered by (tile, cell, class)."""
    prm = SCENES[scene]
    K = prm["classes"]
    p = pts.double()
    Tt = torch.from_numpy(T).to(DEV)
    rng_ = (p[:, 0] * p[:, 0] + p[:, 1] * p[:, 1] + p[:, 2] * p[:, 2]).sqrt()
    ok = (rng_ >= prm["min_range"]) & (rng_ <= prm["max_range"])
    p, lab = p[ok], lab[ok].long()
    w = torch.stack([((p[:, 0] * Tt[r, 0] + p[:, 1] * Tt[r, 1]) + p[:, 2] * Tt[r, 2]) + Tt[r, 3] for r in range(3)], 1)
    w = w.float()
    o = Tt[:3, 3].float()
    e = w - o
    r = torch.sqrt((e[:, 0] * e[:, 0] + e[:, 1] * e[:, 1]) + e[:, 2] * e[:, 2])
    s = torch.full_like(r, prm["free_step"])
    n = torch.floor(r / s)
    for _ in range(2):
        n = torch.where(n * s < r, n, n - 1).clamp(min=0)
    for _ in range(2):
        n = torch.where((n + 1) * s < r, n + 1, n)
    n = torch.where(r > 0, n, 0).long()
    beam = torch.repeat_interleave(torch.arange(len(n), device=DEV), n)
    j = torch.arange(len(beam), device=DEV) - (n.cumsum(0) - n)[beam] + 1
    t = r[beam] - j.float() * s[beam]
    q = t / r[beam]
    free = o + e[beam] * q[:, None]
    x = torch.cat([w, free])
    y = torch.cat([lab if probs is None else probs[ok].argmax(1) + 1, torch.zeros_like(beam)])
    inv = torch.full_like(x, float(np.float32(1.0 / prm["res"])))
    c = torch.floor(x * inv).long()
    lo = c.amin(0) >> 3
    tile, loc = (c >> 3) - lo, c & 7
    ext = tile.amax(0) + 1
    key = (tile[:, 0] * ext[1] + tile[:, 1]) * ext[2] + tile[:, 2]
    key = (key * 512 + (loc[:, 2] * 64 + loc[:, 1] * 8 + loc[:, 0])) * 32 + y
    uniq, idx, cnt = torch.unique(key, return_inverse=True, return_counts=True)
    mean = torch.zeros(len(uniq), 3, device=DEV, dtype=torch.float64).index_add_(0, idx, x.double())
    mean = (mean / cnt[:, None]).float()
    wt = None
    if probs is not None:
        full = torch.zeros(len(x), K + 1, device=DEV, dtype=torch.float64)
        full[:len(w), 1:] = probs[ok].double()
        full[len(w):, 0] = 1.0
        wt = torch.zeros(len(uniq), K + 1, device=DEV, dtype=torch.float64).index_add_(0, idx, full) / cnt[:, None]
    return mean, uniq % 32, wt


def _kernel(r):
    return (2 + torch.cos(2 * math.pi * r)) * (1 - r) / 3 + torch.sin(2 * math.pi * r) / (2 * math.pi)


def _voxels(xyz, res):
    return torch.floor(xyz * torch.full_like(xyz, float(np.float32(1.0 / res)))).long()


class _Field:
    """Eq. (alpha_kernel) on the voxels of a box [lo, lo + ext), by the plain definition."""

    def __init__(self, xyz, res, lmax, edge, lo=None, ext=None):
        self.res, self.R, self.edge = res, int(math.ceil(lmax / res + 0.5)), edge
        self.v, self.x = _voxels(xyz, res), xyz.double()
        self.lo = self.v.amin(0) - self.R if lo is None else torch.tensor(lo, device=DEV)
        self.ext = (self.v.amax(0) + self.R + 1 - self.lo).tolist() if ext is None else ext
        self.size = int(self.ext[0] * self.ext[1] * self.ext[2])

    def at(self, v):
        """Row of each voxel (x fastest), -1 outside the box."""
        g = v - self.lo
        inside = ((g >= 0) & (g < torch.tensor(self.ext, device=DEV))).all(1)
        return torch.where(inside, (g[:, 2] * self.ext[1] + g[:, 1]) * self.ext[0] + g[:, 0], -1)

    def pairs(self, l, face=False):
        """Per candidate offset: (points i, rows, c - x, d) of the pairs within l (one, or one per point)."""
        R = self.R
        for dz in range(-R, R + 1):
            for dy in range(-R, R + 1):
                for dx in range(-R, R + 1):
                    if max(abs(dx) - 1, 0) ** 2 + max(abs(dy) - 1, 0) ** 2 + max(abs(dz) - 1, 0) ** 2 > R * R:
                        continue
                    c = self.v + torch.tensor([dx, dy, dz], device=DEV)
                    e = (c.double() + 0.5) * self.res - self.x
                    d = (e * e).sum(1).sqrt()
                    row = self.at(c)
                    m = (d < l) & (row >= 0)
                    if face:
                        m &= ((c // self.edge) - (self.v // self.edge)).abs().sum(1) <= 1
                    i = m.nonzero()[:, 0]
                    yield i, row[i], e[i], d[i]


def _l_scale(case, K):
    return [L_SCALES[k % len(L_SCALES)] if case.get("form") == "scales" else 1.0 for k in range(K + 1)]


def _alpha(field, cls, wt, K, l, sigma0, face=False, count=False):
    """alpha [rows of the box, K+1] (64 bits); l: one, or one per point."""
    a = torch.full((field.size * (K + 1),), ALPHA0, device=DEV, dtype=torch.float64)
    if count:
        row = field.at(field.v)
        i = (row >= 0).nonzero()[:, 0]
        return a.index_add_(0, row[i] * (K + 1) + cls[i], torch.ones_like(i, dtype=torch.float64)).view(-1, K + 1)
    for i, row, _, d in field.pairs(l, face):
        k = sigma0 * _kernel(d / (l[i] if torch.is_tensor(l) else l))
        if wt is None:
            a.index_add_(0, row * (K + 1) + cls[i], k)
        else:
            a.view(-1, K + 1).index_add_(0, row, k[:, None] * wt[i])
    return a.view(-1, K + 1)


def _mean_var(a):
    S = a.sum(1, keepdim=True)
    return a / S, a * (S - a) / (S * S * (S + 1))


# ---------------------------------------------------------------- inputs of a case
def _inputs(case, seed):
    """Scans of a case, with softmax rows where the form wants them."""
    kind, scene = case["kind"], case["scene"]
    keep = _batch_sizes(case, seed) if kind == "batch" else None
    scans = _scans(scene, case.get("rays", 131072), case.get("scans", case.get("maps", 1)), seed, keep)
    probs = None
    if case.get("form") == "soft":
        gen = torch.Generator(device=DEV)
        gen.manual_seed(seed + 1)
        lab = scans[0][1]
        z = 1.5 * torch.randn(len(lab), SCENES[scene]["classes"], generator=gen, device=DEV)
        z[torch.arange(len(lab), device=DEV), lab.long() - 1] += 5.0
        probs = torch.softmax(z, 1).contiguous()
    return scans, probs


def _params(case, **kw):
    prm = SCENES[case["scene"]]
    return sb.default_params(res=prm["res"], length_scale=case["lr"] * prm["res"], sigma0=prm["sigma0"], alpha0=ALPHA0,
                             free_step=prm["free_step"], num_classes=prm["classes"], min_range=prm["min_range"],
                             max_range=prm["max_range"], block_edge=case.get("edge", 8), **kw)


def _window(case, T):
    """(lowest voxel, extent) of the window read around a sensor, and its voxel centres, x fastest."""
    res, n, h = SCENES[case["scene"]]["res"], case["side"], case["height"]
    lo = [int(math.floor(T[0, 3] / res)) - n // 2, int(math.floor(T[1, 3] / res)) - n // 2,
          int(math.floor(T[2, 3] / res)) - 2 * h // 3]
    z, y, x = torch.meshgrid(*[torch.arange(k, device=DEV, dtype=torch.float64) for k in (h, n, n)], indexing="ij")
    v = torch.stack([x + lo[0], y + lo[1], z + lo[2]], -1).reshape(-1, 3)
    return lo, [n, n, h], ((v + 0.5) * res).float().contiguous()


def _joined(case, scans, probs=None):
    """Training sets of the scans: one each, or all joined (they go into one map)."""
    sets = [_training(case["scene"], *s, probs) for s in scans]
    if case["kind"] in ("stream", "grad", "points"):
        return [(torch.cat([s[0] for s in sets]), torch.cat([s[1] for s in sets]), None)]
    return sets


def _learning(case, train, seed):
    """`points` of a training set (scan after scan) and a tenth as many held-out points near others of it."""
    xyz, cls, _ = train
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed + 2)
    pick = torch.randint(0, len(xyz), (case["points"],), generator=gen, device=DEV).sort().values
    near = torch.randint(0, len(xyz), (max(1, case["points"] // 10),), generator=gen, device=DEV)
    h = xyz[near] + 0.02 * torch.randn(len(near), 3, generator=gen, device=DEV)
    x = xyz[pick] + 0.01 * torch.randn(len(pick), 3, generator=gen, device=DEV)
    return x.contiguous(), cls[pick], h.contiguous(), cls[near].to(torch.int32).contiguous()


def _query_points(xyz, queries, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed + 3)
    at = torch.randint(0, len(xyz), (queries,), generator=gen, device=DEV)
    return (xyz[at] + 0.15 * torch.randn(queries, 3, generator=gen, device=DEV)).contiguous()


def _snapshot(case, seed):
    """Voxel keys and alpha of a mapped window (layers near the ground mapped, some blocks never reached), and the
    world points read."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    n, h, K1 = case["extent"], case["height"], case["classes"] + 1
    z, y, x = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(n, device=DEV), torch.arange(n, device=DEV),
                             indexing="ij")
    keys = torch.stack([x - n // 2, y - n // 2, z - 4], -1).reshape(-1, 3)
    block = torch.rand((h + 16) // 8 * ((n + 16) // 8) ** 2, generator=gen, device=DEV)
    b = (keys + torch.tensor([n // 2 + 8, n // 2 + 8, 4], device=DEV)) // 8
    mapped = block[((b[:, 2] * ((n + 16) // 8) + b[:, 1]) * ((n + 16) // 8) + b[:, 0]) % len(block)] < 0.85
    main = torch.randint(0, K1, (len(keys),), generator=gen, device=DEV)
    main = torch.where(torch.rand(len(keys), generator=gen, device=DEV) < 0.7, 0, main)  # mostly free space
    a = 0.05 * torch.rand(len(keys), K1, generator=gen, device=DEV) ** 4
    a[torch.arange(len(keys), device=DEV), main] += 20.0 * torch.rand(len(keys), generator=gen, device=DEV)
    few = torch.rand(len(keys), generator=gen, device=DEV) < 0.05
    a[few] += 1.5  # voxels with mass in every class: the mode exists
    alpha = (a + ALPHA0).float()
    pts = (keys.double() + 0.5) * 0.1
    if case["order"] == "cloud":  # a point cloud's order and positions inside the voxels
        perm = torch.randperm(len(keys), generator=gen, device=DEV)
        pts = pts[perm] + 0.09 * (torch.rand(len(keys), 3, generator=gen, device=DEV, dtype=torch.float64) - 0.5)
    return keys[mapped].contiguous(), alpha[mapped].contiguous(), pts.float().contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "readoff":
        keys, alpha, pts = _snapshot(case, seed)
        m = sb.Map(sb.default_params(num_classes=case["classes"], pool_blocks=1 << 15, sample_capacity=1 << 16))
        m.import_(keys, alpha)
        q, K1 = len(pts), case["classes"] + 1
        rows = lambda: torch.empty(q, K1, device=DEV)  # noqa: E731
        ints = lambda: torch.empty(q, device=DEV, dtype=torch.int32)  # noqa: E731
        out = dict(probs=rows(), var=rows(), mode=rows(), p_occ=torch.empty(q, device=DEV), label=ints(), state=ints())
        return dict(kind=kind, m=m, pts=pts, out=out)
    scans, probs = _inputs(case, seed)
    if kind == "train":
        return dict(kind=kind, params=_params(case), scan=scans[0], out=torch.zeros(131072, 4, device=DEV))
    if kind == "points":
        xyz, cls, _ = _joined(case, scans)[0]
        return dict(kind=kind, params=_params(case), xyzl=torch.cat([xyz, cls[:, None].float()], 1).contiguous(),
                    pts=_query_points(xyz, case["queries"], seed))
    if kind == "grad":
        xyz, cls, h, hl = _learning(case, _joined(case, scans)[0], seed)
        m = sb.Map(_params(case, pool_blocks=1 << 14, sample_capacity=1 << 23))
        return dict(kind=kind, m=m, xyz=xyz, cls=cls.to(torch.int32), h=h, hl=hl,
                    xyzl=torch.cat([xyz, cls[:, None].float()], 1).contiguous())
    form = case.get("form", "hard")
    K = SCENES[case["scene"]]["classes"]
    kw = dict(pool_blocks=1 << 16, sample_capacity=1 << 24)
    if kind == "batch":
        kw = dict(pool_blocks=1 << 18, sample_capacity=1 << 26, num_maps=case["maps"])
    if form == "count":
        kw["sensor_model"] = 1
    if form == "face":
        kw["association"] = 1
    if form == "scales":
        kw["l_scale"] = _l_scale(case, K)
    m = sb.Map(_params(case, **kw))
    # a stream is read around its last pose
    centres = [_window(case, T)[2] for _, _, T in (scans[-1:] if kind == "stream" else scans)]
    if case.get("host"):
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        scans = [(pin(p), pin(l), T) for p, l, T in scans]
        probs = pin(probs) if probs is not None else None
    reads = [(c, torch.empty(len(c), K + 1, device=DEV), torch.empty(len(c), K + 1, device=DEV)) for c in centres]
    batch = None
    if kind == "batch":
        batch = [dict(points=p, labels=l, pose=T, map_id=i) for i, (p, l, T) in enumerate(scans)]
    return dict(kind=kind, m=m, scans=scans, probs=probs, reads=reads, batch=batch)


STATS = ("hits", "dropped", "free_samples", "train_points", "touched_blocks", "pairs", "total_blocks")


def run(s):
    kind = s["kind"]
    if kind == "train":
        pts, lab, T = s["scan"]
        n = sb.training_set_noalloc(s["params"], pts, lab, T, s["out"])
        return [s["out"], n]
    if kind == "points":
        return sb.query_points(s["params"], s["xyzl"], s["pts"])
    m = s["m"]
    if kind == "readoff":
        m.query_device(s["pts"], **s["out"])
        return dict(s["out"])
    if kind == "grad":
        st = m.insert_training(s["xyz"], s["cls"])
        m.grad_clear()
        ll = m.heldout_loglik(s["h"], s["hl"], grad=True)
        gl, gs, gx = m.backward(s["xyzl"])
        return dict(ll=ll, grad_l=gl, grad_sigma0=gs, grad_xyz=gx, stats=[st["pairs"], st["touched_blocks"]])
    if kind == "batch":
        st = m.insert_batch(s["batch"])
    elif kind == "stream":
        for pts, lab, T in s["scans"]:
            m.insert_scan(pts, lab, T, sync=False)
        st = m.sync()
    elif s["probs"] is not None:
        pts, _, T = s["scans"][0]
        st = m.insert_scan_soft(pts, s["probs"], T)
    else:
        pts, lab, T = s["scans"][0]
        st = m.insert_scan(pts, lab, T)
    for i, (centres, mean, var) in enumerate(s["reads"]):
        if kind == "batch":
            m.select(i)
        m.query_device(centres, mean, var=var)
    return dict(read=[[mean, var] for _, mean, var in s["reads"]], stats=[st[k] for k in STATS])


def work(case):
    """Bytes: inputs and outputs once, and a read and a write of the increments that the pass adds to (about 18 voxels
    and 6 training points per ray of a LiDAR, 1.5 and 1 of a depth image; one class each).  Operations: about 30 per
    pair of a voxel and a training point within l."""
    kind = case["kind"]
    if kind == "readoff":
        q, K1 = case["extent"] ** 2 * case["height"], case["classes"] + 1
        return {"bytes": q * (12.0 + 4 * K1 + 12 * K1 + 12), "flops": 12.0 * q * K1}
    K1 = SCENES[case["scene"]]["classes"] + 1
    ball = 4.19 * case["lr"] ** 3
    if kind == "batch":
        hits = float(sum(_batch_sizes(case, 0)))
    else:
        hits = float(case.get("points", case.get("rays", 0))) * (case.get("scans", 1) if kind == "stream" else 1)
    room = case["scene"] == "room"
    points, voxels = (1.0 if room else 6.0) * hits, (1.5 if room else 18.0) * hits
    if kind == "train":
        return {"bytes": 16.0 * hits + 16 * points, "flops": 30.0 * points}
    if kind == "points":
        return {"bytes": 16.0 * points + case["queries"] * (12.0 + 4 * K1), "flops": 12.0 * case["queries"] * ball}
    if kind == "grad":
        return {"bytes": hits * (16 + 16 + 12) + 8.0 * hits + 1.6 * hits, "flops": 70.0 * hits * ball}
    read = case["side"] ** 2 * case["height"] * (12.0 + 12 * K1) * case.get("maps", 1)
    per_hit = 12.0 + 4 * (K1 - 1) if case.get("form") == "soft" else 16.0
    if case.get("form") == "count":
        return {"bytes": per_hit * hits + 8 * points + read, "flops": 30.0 * points}
    return {"bytes": per_hit * hits + 8.0 * voxels + read, "flops": 30.0 * points * ball}


# ---------------------------------------------------------------- the definition in 64 bits
def exact(case, seed):
    kind = case["kind"]
    if kind == "readoff":
        return _exact_readoff(case, seed)
    prm = SCENES[case["scene"]]
    K, l = prm["classes"], case["lr"] * prm["res"]
    scans, probs = _inputs(case, seed)
    sets = _joined(case, scans, probs)
    if kind == "train":
        xyz, cls, _ = sets[0]
        out = torch.zeros(131072, 4, device=DEV, dtype=torch.float64)
        out[:len(xyz)] = torch.cat([xyz, cls[:, None].float()], 1)
        return [out, None]
    if kind == "points":
        return _exact_points(sets[0], _query_points(sets[0][0], case["queries"], seed), K, l, prm)
    if kind == "grad":
        return _exact_grad(*_learning(case, sets[0], seed), K, l, prm)
    ls = torch.tensor(_l_scale(case, K), device=DEV, dtype=torch.float64) * l
    read = []
    for (xyz, cls, wt), (_, _, T) in zip(sets, scans[-1:] if kind == "stream" else scans):
        lo, ext, _ = _window(case, T)
        f = _Field(xyz, prm["res"], float(ls.max()), case.get("edge", 8), lo, ext)
        a = _alpha(f, cls, wt, K, ls[cls] if case.get("form") == "scales" else l, prm["sigma0"],
                   case.get("form") == "face", case.get("form") == "count")
        read.append(list(_mean_var(a)))
    return dict(read=read, stats=[None] * len(STATS))


def _exact_readoff(case, seed):
    keys, alpha, pts = _snapshot(case, seed)
    K1 = case["classes"] + 1
    a0 = torch.tensor(ALPHA0, device=DEV, dtype=torch.float32)
    lo = keys.amin(0)
    ext = keys.amax(0) - lo + 1
    row = torch.full((int(ext[0] * ext[1] * ext[2]),), -1, dtype=torch.int64, device=DEV)
    k = keys - lo
    row[(k[:, 2] * ext[1] + k[:, 1]) * ext[0] + k[:, 0]] = torch.arange(len(k), device=DEV)
    v = torch.floor(pts * torch.full_like(pts, 10.0)).long() - lo
    inside = ((v >= 0) & (v < ext)).all(1)
    r = torch.where(inside, row[((v[:, 2] * ext[1] + v[:, 1]) * ext[0] + v[:, 0]).clamp(0, len(row) - 1)], -1)
    inc = torch.where((r >= 0)[:, None], (alpha - a0)[r.clamp(min=0)], torch.zeros((), device=DEV))
    a = (a0 + inc).double()
    S = a.sum(1, keepdim=True)
    mean, var = _mean_var(a)
    mode = torch.where((a > 1).all(1, keepdim=True), (a - 1) / (S - K1), math.nan)
    return dict(probs=mean, var=var, mode=mode, p_occ=mean[:, 1:].sum(1), label=None, state=None)


def _exact_points(train, pts, K, l, prm):
    """Cells of edge res; the cells of each query's neighbourhood, run by run."""
    xyz, cls, _ = train
    res, R = prm["res"], int(math.ceil(l / prm["res"])) + 1
    c = torch.floor(xyz.double() / res).long()
    lo = c.amin(0) - 1
    ext = c.amax(0) + 2 - lo
    flat = lambda v: (v[:, 2] * ext[1] + v[:, 1]) * ext[0] + v[:, 0]  # noqa: E731
    f, order = flat(c - lo).sort()
    x, y = xyz.double()[order], cls[order]
    size = int(ext[0] * ext[1] * ext[2])
    count = torch.bincount(f, minlength=size)
    start = count.cumsum(0) - count
    cq, pq = torch.floor(pts.double() / res).long(), pts.double()
    a = torch.full((len(pts), K + 1), ALPHA0, device=DEV, dtype=torch.float64)
    for dz in range(-R, R + 1):
        for dy in range(-R, R + 1):
            for dx in range(-R, R + 1):
                v = cq + torch.tensor([dx, dy, dz], device=DEV) - lo
                at = torch.where(((v >= 0) & (v < ext)).all(1), flat(v), -1)
                n = torch.where(at >= 0, count[at.clamp(min=0)], 0)
                i = (n > 0).nonzero()[:, 0]
                j = 0
                while len(i):
                    t = start[at[i]] + j
                    d = (pq[i] - x[t]).norm(dim=1)
                    k = torch.where(d < l, prm["sigma0"] * _kernel(d / l), 0.0)
                    a.index_put_((i, y[t]), k, accumulate=True)
                    j += 1
                    i = i[n[i] > j]
    return a


def _exact_grad(xyz, cls, h, hl, K, l, prm):
    sigma0, hl = prm["sigma0"], hl.long()
    f = _Field(xyz, prm["res"], l, 8)
    a = _alpha(f, cls, None, K, l, sigma0)
    r = f.at(_voxels(h, prm["res"]))
    ok = r >= 0
    S = torch.where(ok, a.sum(1)[r.clamp(min=0)], ALPHA0 * (K + 1))
    ay = torch.where(ok, a[r.clamp(min=0), hl], ALPHA0)
    ll = torch.log(ay / S).sum()
    G = torch.zeros_like(a)
    G.index_add_(0, r[ok], (-1.0 / S[ok])[:, None].expand(-1, K + 1).contiguous())
    G.index_put_((r[ok], hl[ok]), 1.0 / ay[ok], accumulate=True)
    gx = torch.zeros(len(xyz), 3, device=DEV, dtype=torch.float64)
    gl, gs = torch.zeros((), device=DEV, dtype=torch.float64), torch.zeros((), device=DEV, dtype=torch.float64)
    for i, row, e, d in f.pairs(l):
        u = d / l
        g = G[row, cls[i]]
        # f'(r) = -(2/3) (pi (1 - r) sin(2 pi r) + 1 - cos(2 pi r))
        df = -(2.0 / 3.0) * (math.pi * (1 - u) * torch.sin(2 * math.pi * u) + 1 - torch.cos(2 * math.pi * u))
        gs += (g * _kernel(u)).sum()
        gl += (g * sigma0 * df * (-d / (l * l))).sum()
        gx[i] += (g * sigma0 * df / (l * d.clamp(min=1e-300)))[:, None] * -e
    return dict(ll=ll, grad_l=gl, grad_sigma0=gs, grad_xyz=gx, stats=[None, None])
