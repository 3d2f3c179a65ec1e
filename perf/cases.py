"""Performance cases of the kmx front end.

Each case is a piece of work that a user of the library gives it, at a size that
the repository's own configurations, benchmark or tests use: the stages of one
cloud (voxelise, ground suppression, descriptors), descriptor matching in both
modes, registration from correspondences, and whole pairs.

Clouds are drawn on the GPU from a seed: a ray-cast street scene (64-beam
scanner), a furnished room and a 10 m cube with planes, spheres and cylinders.
Descriptors that only feed a matching case come from a plain FP64 chain in this
file with order-independent sums, so they depend on the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")
F64 = torch.float64
EXACT_PAIRS = 1e11  # descriptor pairs beyond which no 64-bit matching is formed


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # a small scan joining a batch (the batches start at 5k points): launches count
        dict(name="voxelize_scene_6k", op="voxelize", kind="cube", n=6001, voxel=0.1, stride=3, assign=False),
        # one cloud of the large dense indoor pair, with the point-to-voxel map
        dict(name="voxelize_room_2M", op="voxelize", kind="room", n=2000000, voxel=0.02, stride=3, assign=True),
        # geometric suppression of one scan (64 beams, 2048 azimuth bins)
        dict(name="ground_lidar_121k", op="ground", n=121003, stride=3),
        # grid, normals and Faster-PFH of one scan
        dict(name="features_lidar_19k", op="features", kind="lidar", n=18755, method="lists"),
        # the same of one cloud of the large dense indoor pair
        dict(name="features_room_300k", op="features", kind="room", n=300017, method="lists"),
        # a small pair's matching: the smallest calls, where launches count
        dict(name="match_exact_1k", op="match", mode="fp32", kind="cube", n_src=1021, n_tgt=897),
        # one scan pair's matching (12.8k reliable descriptors a side)
        dict(name="match_exact_13k", op="match", mode="fp32", kind="lidar", n_src=12778, n_tgt=12776),
        # a query scan against a resident map, and the larger members of a batch
        dict(name="match_tensor_40k", op="match", mode="bf16", kind="room", n_src=40009, n_tgt=61003),
        # matching of the large dense indoor pair
        dict(name="match_tensor_300k", op="match", mode="bf16", kind="room", n_src=302548, n_tgt=287858),
        # correspondences to pose: ratio filter, k-core, GNC, on one scan pair's matches
        dict(name="register_5k", op="register", n=4778, n_tau=3000),
        # a whole scan pair, replayed as the graph that a streaming user keeps
        dict(name="pair_lidar_121k", op="pair", kind="lidar", n_src=121003, n_tgt=120501, voxel=0.3, mode="fp32",
             suppress=False),
        # the whole large dense indoor pair, the benchmark's headline workload
        dict(name="pair_room_2M", op="pair", kind="room", n_src=2000000, n_tgt=2000000, voxel=0.02, mode="bf16",
             suppress=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["voxelize", "ground", "features", "features", "match", "match", "match", "register", "pair"])
    if op == "voxelize":
        kind = rng.choice(["cube", "lidar", "room"])
        n = _log_int(rng, 5000, 2000000)
        voxel = rng.choice([0.02, 0.05]) if kind == "room" else rng.choice([0.05, 0.1, 0.3])
        return dict(op=op, kind=kind, n=n, voxel=voxel, stride=rng.choice([3, 4]), assign=rng.random() < 0.5)
    if op == "ground":
        return dict(op=op, n=_log_int(rng, 20000, 250000), stride=rng.choice([3, 4]))
    if op == "features":
        kind = rng.choice(["cube", "lidar", "room"])
        hi = 300000 if kind == "room" else 60000
        return dict(op=op, kind=kind, n=_log_int(rng, 2000, hi), method=rng.choice(["lists", "lists", "faster"]))
    if op == "match":
        mode = rng.choice(["fp32", "bf16"])
        lo, hi = (300, 16000) if mode == "fp32" else (15000, 290000)
        kind = rng.choice(["cube", "lidar"]) if mode == "fp32" else "room"
        n = _log_int(rng, lo, hi)
        return dict(op=op, mode=mode, kind=kind, n_src=n, n_tgt=max(lo, min(hi, int(n * rng.uniform(0.5, 1.5)))))
    if op == "register":
        return dict(op=op, n=_log_int(rng, 600, 30000), n_tau=rng.choice([1000, 3000, 4096]))
    kind = rng.choice(["cube", "lidar", "room"])
    n = _log_int(rng, 5000, 300000)
    return dict(op=op, kind=kind, n_src=n, n_tgt=int(n * rng.uniform(0.7, 1.0)),
                voxel=0.3 if kind == "lidar" else rng.choice([0.05, 0.1]), mode="bf16" if n > 200000 else "fp32",
                suppress=kind == "lidar" and rng.random() < 0.5)


def _neighbours(kind):
    """Mean r_FPFH neighbours of a voxel, including itself."""
    return {"cube": 145, "lidar": 41, "room": 166}[kind]


def _feature_work(kind, n, lists):
    # a distance test per neighbour and covariance terms (25), one pair feature (70)
    # and one histogram row added (66) each; rows, normals and lists written once
    m = _neighbours(kind)
    return n * (16 + 16 + 1 + 144 + 4 + (8 + 4 * m if lists else 0)), n * m * 161.0


def work(case):
    op = case["op"]
    if op == "voxelize":
        n = case["n"]
        return {"bytes": n * (4 * case["stride"] + (4 if case["assign"] else 0)) + 16 * (n // 6), "flops": 6.0 * n}
    if op == "ground":
        n = case["n"]
        return {"bytes": 4 * case["stride"] * n * 1.13, "flops": 60.0 * n}
    if op == "features":
        b, f = _feature_work(case["kind"], case["n"], case["method"] == "lists")
        return {"bytes": b, "flops": f}
    if op == "match":
        ns, nt = case["n_src"], case["n_tgt"]
        return {"bytes": (ns + nt) * 148 + 16 * (min(ns, nt) // 3), "flops": 66.0 * ns * nt}
    if op == "register":
        k = min(case["n"], case["n_tau"])
        return {"bytes": 16 * case["n"] + 32 * k, "flops": 10.0 * k * k + 44 * 80.0 * k}
    ns, nt = case["n_src"] // 6, case["n_tgt"] // 6
    bs, fs = _feature_work(case["kind"], ns, False)
    bt, ft = _feature_work(case["kind"], nt, False)
    return {"bytes": 12 * (case["n_src"] + case["n_tgt"]) + bs + bt + 16 * min(ns, nt) // 3,
            "flops": fs + ft + 66.0 * ns * nt}


# ---------------------------------------------------------------------------
# seeded clouds
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=F64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=F64)


def _box_faces(lo, hi):
    e = np.diag(np.asarray(hi, float) - np.asarray(lo, float))
    lo = np.asarray(lo, float)
    return [(lo + s * e[c], e[a], e[b]) for a, b, c in ((0, 1, 2), (0, 2, 1), (1, 2, 0)) for s in (0, 1)]


def _scene(kind, rng):
    """(parallelograms [o, e1, e2], upright cylinders [base, r, h], spheres [c, r], viewpoint, noise)."""
    rects, cyls, balls = [], [], []
    x, y, z = np.eye(3)
    if kind == "cube":
        rects = [(0 * x, 10 * x, 10 * y), (0 * x, 10 * y, 10 * z), (0 * x, 10 * x, 10 * z)]
        for _ in range(4):
            r = rng.uniform(0.3, 1.0)
            balls.append((np.array([rng.uniform(1.5, 8.5), rng.uniform(1.5, 8.5), rng.uniform(r + 0.5, 6)]), r))
        for _ in range(3):
            cyls.append((np.array([rng.uniform(1, 9), rng.uniform(1, 9), 0]), rng.uniform(0.2, 0.5), rng.uniform(1, 4)))
        return rects, cyls, balls, np.array([5.0, 5.0, 5.0]), 0.01
    w, d, h = 4.0, 3.0, 2.2
    rects = [(0 * x, w * x, d * y), (0 * x, w * x, h * z), (d * y, w * x, h * z), (0 * x, d * y, h * z),
             (w * x, d * y, h * z)]
    for _ in range(40):
        s = np.array([rng.uniform(0.1, 0.4), rng.uniform(0.1, 0.4), rng.uniform(0.15, 0.6)])
        o = np.array([rng.uniform(0.1, w - s[0] - 0.1), rng.uniform(0.1, d - s[1] - 0.1), 0])
        rects += _box_faces(o, o + s)
        cyls.append((o + s * [0.5, 0.5, 1], rng.uniform(0.02, 0.08), rng.uniform(0.15, 0.5)))
    return rects, cyls, balls, np.array([2.0, 1.5, 1.1]), 0.005


def _surface_cloud(kind, n, scene_seed, g):
    """n noisy samples of the scene's surfaces, uniform by area, FP64."""
    rects, cyls, balls, vp, noise = _scene(kind, np.random.default_rng(scene_seed))
    row = [np.concatenate(r) for r in rects]
    row += [np.concatenate([c, [r, h, 0], [0, 0, 0]]) for c, r, h in cyls]
    row += [np.concatenate([c, [r, 0, 0], [0, 0, 0]]) for c, r in balls]
    area = [np.linalg.norm(a) * np.linalg.norm(b) for _, a, b in rects]
    area += [2 * math.pi * r * h for _, r, h in cyls] + [4 * math.pi * r * r for _, r in balls]
    edge = torch.tensor(np.cumsum(area) / np.sum(area), device=DEV)
    edge[-1] = 2.0
    which = torch.searchsorted(edge, _rand(g, n), right=True)
    t = torch.tensor(np.array(row), device=DEV)[which]
    u = _rand(g, n, 2)
    o, a, b = t[:, 0:3], t[:, 3:6], t[:, 6:9]
    phi = 2 * math.pi * u[:, 0]
    c, s = torch.cos(phi), torch.sin(phi)
    side = torch.stack([a[:, 0] * c, a[:, 0] * s, a[:, 1] * u[:, 1]], 1)
    zz = 2 * u[:, 1] - 1
    rho = torch.sqrt((1 - zz * zz).clamp_min(0))
    ball = a[:, :1] * torch.stack([rho * c, rho * s, zz], 1)
    p = torch.where((which < len(rects))[:, None], u[:, :1] * a + u[:, 1:] * b,
                    torch.where((which < len(rects) + len(cyls))[:, None], side, ball))
    return o + p + noise * _randn(g, n, 3), vp


def _scan(n, scene_seed, view, g):
    """n returns, in scan order, of a 64-beam scanner in a street scene (ground,
    30 boxes, 10 walls, 50 poles), FP64 in the sensor's frame; view 1 stands 10 m
    further on and is turned."""
    rng = np.random.default_rng(scene_seed)
    boxes, poles = [], []
    while len(boxes) < 40:
        wall = len(boxes) >= 30
        hx, hy = (rng.uniform(5, 20), 0.15) if wall else rng.uniform(0.5, 2.5, 2)
        cx, cy = rng.uniform(-70, 70, 2)
        if not (-8 - hx < cx < 18 + hx and abs(cy) < 4 + hx):
            boxes.append((cx, cy, rng.uniform(0, math.pi), hx, hy, rng.uniform(3, 6) if wall else rng.uniform(1, 4)))
    while len(poles) < 50:
        cx, cy = rng.uniform(-70, 70, 2)
        if not (-8 < cx < 18 and abs(cy) < 4.5):
            poles.append((cx, cy, rng.uniform(0.1, 0.3), rng.uniform(3, 8)))
    yaw = math.radians(rng.uniform(-30, 30)) if view else 0.0
    org = (10.0, 0.0, 1.73) if view else (0.0, 0.0, 1.73)
    bx = torch.tensor(np.array(boxes), device=DEV)
    po = torch.tensor(np.array(poles), device=DEV)
    inf = float("inf")
    bins = int(n / 64 / 0.95) + 1
    while True:
        elev = torch.deg2rad(torch.linspace(-25.0, 3.0, 64, dtype=F64, device=DEV))
        az = 2 * math.pi * (torch.arange(bins, dtype=F64, device=DEV) + 0.5) / bins
        e, a = torch.meshgrid(elev, az, indexing="ij")
        ds = torch.stack([torch.cos(e) * torch.cos(a), torch.cos(e) * torch.sin(a), torch.sin(e)], -1).reshape(-1, 3)
        c, s = math.cos(yaw), math.sin(yaw)
        d = torch.stack([c * ds[:, 0] - s * ds[:, 1], s * ds[:, 0] + c * ds[:, 1], ds[:, 2]], 1)
        hit = torch.empty(len(d), dtype=F64, device=DEV)
        for k in range(0, len(d), 1 << 18):
            q = d[k:k + (1 << 18)]
            best = torch.where(q[:, 2] < -1e-9, -org[2] / q[:, 2], inf)
            cy, sy = torch.cos(bx[:, 2]), torch.sin(bx[:, 2])
            ox, oy = org[0] - bx[:, 0], org[1] - bx[:, 1]
            lo, hi = torch.zeros(len(q), len(bx), dtype=F64, device=DEV), inf
            for p, v, a0, a1 in ((cy * ox + sy * oy, q[:, :1] * cy + q[:, 1:2] * sy, -bx[:, 3], bx[:, 3]),
                                 (cy * oy - sy * ox, q[:, 1:2] * cy - q[:, :1] * sy, -bx[:, 4], bx[:, 4]),
                                 (torch.full_like(ox, org[2]), q[:, 2:3].expand(-1, len(bx)), 0 * bx[:, 5], bx[:, 5])):
                v = torch.where(v.abs() < 1e-12, 1e-12, v)
                t0, t1 = (a0 - p) / v, (a1 - p) / v
                lo = torch.maximum(lo, torch.minimum(t0, t1))
                hi = torch.maximum(t0, t1) if isinstance(hi, float) else torch.minimum(hi, torch.maximum(t0, t1))
            best = torch.minimum(best, torch.where((hi >= lo) & (lo > 1e-6), lo, inf).amin(1))
            ox, oy = org[0] - po[:, 0], org[1] - po[:, 1]
            aa = (q[:, 0] ** 2 + q[:, 1] ** 2)[:, None]
            bb = q[:, :1] * ox + q[:, 1:2] * oy
            disc = bb * bb - aa * (ox * ox + oy * oy - po[:, 2] ** 2)
            tc = (-bb - torch.sqrt(disc.clamp_min(0))) / aa
            z = org[2] + tc * q[:, 2:3]
            best = torch.minimum(best, torch.where((disc >= 0) & (tc > 1e-6) & (z >= 0) & (z <= po[:, 3]), tc, inf).amin(1))
            hit[k:k + (1 << 18)] = best
        ok = torch.nonzero(hit <= 80.0).squeeze(1)
        if len(ok) >= n:
            break
        bins = int(bins * max(1.02, 1.01 * n / max(len(ok), 1))) + 1
    if len(ok) > n:
        ok = ok[torch.randperm(len(ok), generator=g, device=DEV)[:n].sort().values]
    return ds[ok] * (hit[ok] + 0.02 * _randn(g, n))[:, None], np.zeros(3)


def _motion(rng):
    q = rng.standard_normal(4)
    w, x, y, z = q / np.linalg.norm(q)
    R = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                  [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                  [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]])
    return R, rng.uniform(-1, 1, 3)


def _cloud(kind, n, seed, view=0):
    """Raw cloud [n, 3] float32 and its viewpoint; view 1 is a second, moved look at the same scene."""
    g = _gen(2 * seed + view)
    if kind == "lidar":
        p, vp = _scan(n, seed, view, g)
        return p.float(), vp
    p, vp = _surface_cloud(kind, n, seed, g)
    if view:
        R, t = _motion(np.random.default_rng(seed + 7))
        p, vp = p @ torch.tensor(R.T, device=DEV) + torch.tensor(t, device=DEV), R @ vp + t
    return p.float(), vp


def _strided(xyz, stride):
    return xyz.contiguous() if stride == 3 else torch.nn.functional.pad(xyz, (0, 1)).contiguous()


# ---------------------------------------------------------------------------
# the same quantities in plain FP64
# ---------------------------------------------------------------------------

def _sums(x, lengths):
    """Sums of consecutive rows of x, in their order."""
    return torch.segment_reduce(x, "sum", lengths=lengths, axis=0, unsafe=True)


def _voxels64(xyz, voxel):
    """Centroids of the occupied voxels in order of their first point, FP64."""
    v = float(np.float32(voxel))
    k = torch.floor(xyz[:, :3].double() / v).long() + (1 << 20)
    key = (k[:, 0] << 42) | (k[:, 1] << 21) | k[:, 2]
    uniq, inv, cnt = torch.unique(key, return_inverse=True, return_counts=True)
    first = torch.full((len(uniq),), len(key), dtype=torch.long, device=DEV)
    first.scatter_reduce_(0, inv, torch.arange(len(key), device=DEV), "amin")
    rank = torch.empty_like(first)
    rank[torch.argsort(first)] = torch.arange(len(uniq), device=DEV)
    num = torch.empty_like(cnt)
    num[rank] = cnt
    order = torch.argsort(rank[inv], stable=True)
    return _sums(xyz[order, :3].double(), num) / num[:, None]


def _voxel_cloud(kind, n, seed, view=0):
    """n voxelised points [n, 3] float32 of a cloud with the usual 6.5 raw points a
    voxel, the voxel size (float32) that gives them, and the viewpoint."""
    ref, count, power = {"cube": (0.1, 17e3, 2.0), "lidar": (0.3, 18.8e3, 1.2), "room": (0.02, 3e5, 2.0)}[kind]
    raw, vp = _cloud(kind, int(6.5 * n) + 100, seed, view)
    v = ref * (count / n) ** (1 / power)
    for _ in range(40):
        vox = _voxels64(raw, v)
        if n <= len(vox) <= 1.06 * n + 20:
            break
        v *= (len(vox) / (1.03 * n)) ** (1 / power)
    while len(vox) < n:
        v *= 0.97
        vox = _voxels64(raw, v)
    return vox[:n].float(), float(np.float32(v)), vp


def _radius_pairs(p, r):
    """All (q, k) with |p_k - p_q| < r, k = q included, by ascending q, by a sorted 27-cell grid."""
    c = torch.floor(p / (r * (1 + 1e-6))).long() + (1 << 20)
    key = (c[:, 0] << 42) | (c[:, 1] << 21) | c[:, 2]
    key, order = torch.sort(key, stable=True)
    qs, ks = [], []
    for dx in (-1, 0, 1):
        for dy in (-1, 0, 1):
            for dz in (-1, 0, 1):
                want = key + (dx * (1 << 42) + dy * (1 << 21) + dz)
                lo = torch.searchsorted(key, want)
                cnt = torch.searchsorted(key, want, right=True) - lo
                q = torch.repeat_interleave(torch.arange(len(p), device=DEV), cnt)
                at = torch.arange(len(q), device=DEV) - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
                q, k = order[q], order[lo[q] + at]
                ok = ((p[q] - p[k]) ** 2).sum(1) < r * r
                qs.append(q[ok])
                ks.append(k[ok])
    q, order = torch.sort(torch.cat(qs), stable=True)
    return q, torch.cat(ks)[order]


def _normals64(p, q, k, r, vp):
    """Unit normals toward vp and linearity of every point with at least 3 points within r, FP64."""
    n = len(p)
    d = p[k] - p[q]
    near = (d * d).sum(1) < r * r
    q, d = q[near], d[near]
    m = torch.bincount(q, minlength=n)
    d = d - (_sums(d, m) / m[:, None])[q]
    cov = (_sums((d[:, :, None] * d[:, None, :]).reshape(-1, 9), m) / m[:, None]).reshape(n, 3, 3)
    w, v = zip(*(torch.linalg.eigh(cov[s:s + 16384]) for s in range(0, n, 16384)))
    w, v = torch.cat(w), torch.cat(v)
    has = (m >= 3) & (w[:, 2] > 0)
    nv = v[:, :, 0]
    nv = torch.where(((torch.tensor(vp, device=DEV) - p) * nv).sum(1, keepdim=True) < 0, -nv, nv)
    plin = (w[:, 2] - w[:, 1]) / torch.where(has, w[:, 2], 1.0)
    return torch.where(has[:, None], torch.cat([nv, plin[:, None]], 1), 0.0), has


def _descriptors64(xyz, voxel, vp):
    """Faster-PFH in FP64: normals [n, 4], J, and its FPFH rows [|J|, 33]."""
    p, n = xyz[:, :3].double(), len(xyz)
    v = np.float32(voxel)
    r_normal, r_fpfh = float(np.float32(3.5) * v), float(np.float32(5.0) * v)
    q, k = _radius_pairs(p, r_fpfh)
    vp = np.float32(vp).astype(np.float64)
    normal4, has = _normals64(p, q, k, r_normal, vp)
    good = has & (normal4[:, 3] < float(np.float32(0.99))) & (torch.bincount(q, minlength=n) >= 3)
    use = good[q] & good[k]
    q, k = q[use], k[use]
    J = torch.nonzero(good & (torch.bincount(q, minlength=n) >= 3)).squeeze(1)
    use = q != k
    q, k = q[use], k[use]
    # angles of each pair in the Darboux frame of the point whose normal is closer to the line
    d = p[k] - p[q]
    w = torch.sqrt((d * d).sum(1))
    use = w > 0
    q, k, d, w = q[use], k[use], d[use], w[use]
    d = d / w[:, None]
    nq, nk = normal4[q, :3], normal4[k, :3]
    src = ((nq * d).sum(1).abs() >= (nk * d).sum(1).abs())[:, None]
    u, nb = torch.where(src, nq, nk), torch.where(src, nk, nq)
    d = torch.where(src, d, -d)
    x = torch.linalg.cross(d, u)
    s = torch.sqrt((x * x).sum(1))
    x = x / s.clamp_min(1e-300)[:, None]
    y = torch.linalg.cross(u, x)
    f = (torch.atan2((y * nb).sum(1), (u * nb).sum(1)) / math.pi, (x * nb).sum(1), (u * d).sum(1))
    bins = [((a + 1) * 5.5).floor().clamp(0, 10).long() + 11 * i for i, a in enumerate(f)]
    del x, y, u, nb, nq, nk, src, d, f
    use = s >= 1e-6
    hist = torch.zeros(n * 33, dtype=torch.long, device=DEV)
    for b in bins:
        hist += torch.bincount(q[use] * 33 + b[use], minlength=n * 33)
    num = torch.bincount(q[use], minlength=n)
    spfh = hist.reshape(n, 33).double() * (100.0 / num.clamp_min(1).double())[:, None]
    # sums over the neighbours in 2^-30 fixed point: the same in any order
    m = torch.bincount(q, minlength=n).clamp_min(1)
    inv = float(1 << 30) / w
    rows = []
    for h in range(33):
        acc = torch.zeros(n, dtype=torch.long, device=DEV)
        acc.index_add_(0, q, torch.round(spfh[:, h].contiguous()[k] * inv).long())
        rows.append(acc.double() / float(1 << 30) / m)
    return normal4, J, (spfh + torch.stack(rows, 1))[J]


def _rows(kind, n, seed, view):
    """n descriptor rows [n, 36] float32 of a cloud of this kind."""
    size = int(n * (1.7 if kind == "lidar" else 1.02)) + 60
    while True:
        desc = _descriptors64(*_voxel_cloud(kind, size, seed, view))[2]
        if len(desc) >= n:
            return torch.nn.functional.pad(desc[:n].float(), (0, 3)).contiguous()
        size = int(size * 1.15)


def _nearest64(x, y):
    """Per row of x the nearest row of y (lowest on ties), the two smallest distances, and per row of y its
    nearest row of x, FP64."""
    xx, yy = (x * x).sum(1), (y * y).sum(1)
    step = max(1, min(len(x), int(1.5e9 // len(y))))
    near, second = [], []
    best = torch.full((len(y),), float("inf"), dtype=F64, device=DEV)
    back = torch.zeros(len(y), dtype=torch.long, device=DEV)
    for s in range(0, len(x), step):
        d = torch.addmm(yy[None, :], x[s:s + step], y.T, alpha=-2.0) + xx[s:s + step, None]
        a, i = d.min(0)
        back = torch.where(a < best, i + s, back)
        best = torch.minimum(a, best)
        j = d.min(1).indices
        d.scatter_(1, j[:, None], float("inf"))
        near.append(j)
        second.append(d.min(1).indices)
    near, second = torch.cat(near), torch.cat(second)
    dist = [torch.sqrt(((x - y[j]) ** 2).sum(1)) for j in (near, second)]
    return near, dist[0], dist[1], back


# ---------------------------------------------------------------------------
# states
# ---------------------------------------------------------------------------

def _register_problem(case, seed):
    """Matches of a scan pair: a few true ones, many that slid along the ground, the rest at random."""
    g, n = _gen(seed), case["n"]
    src = _voxel_cloud("lidar", n + n // 3, seed)[0]
    a = src[torch.randperm(len(src), generator=g, device=DEV)[:n].sort().values].double()
    R, t = _motion(np.random.default_rng(seed))
    u = _rand(g, n)
    true, slid = u < 0.06, (u >= 0.06) & (u < 0.6)
    slip = 6.0 * _randn(g, n, 3) * torch.tensor([1.0, 1.0, 0.02], device=DEV, dtype=F64)
    move = torch.where(true[:, None], 0.1 * _randn(g, n, 3), slip)
    b = torch.where((true | slid)[:, None], a + move, a[torch.randperm(n, generator=g, device=DEV)])
    b = b @ torch.tensor(R.T, device=DEV) + torch.tensor(t, device=DEV)
    j = torch.randperm(n, generator=g, device=DEV)
    d1 = 60.0 * torch.exp(0.5 * _randn(g, n))
    d2 = d1 * (1.0 + torch.where(true, 0.5, 0.25) * _rand(g, n))
    i = torch.arange(n, device=DEV)
    corr = torch.stack([i.int(), j.int(), d1.float().view(torch.int32), d2.float().view(torch.int32)], 1).contiguous()
    tgt = torch.empty(n, 3, dtype=torch.float32, device=DEV)
    tgt[j] = b.float()
    return corr, _strided(a.float(), 4), _strided(tgt, 4), 0.45


def prepare(case, seed):
    from paper_2409_15615_gb300 import kmx, pipeline

    op = case["op"]
    zeros = lambda *s, dtype=torch.float32: torch.zeros(*s, dtype=dtype, device=DEV)  # noqa: E731
    ctx = kmx.Context(0)
    st = dict(op=op, case=case, ctx=ctx)
    if op == "voxelize":
        n = case["n"]
        st.update(xyz=_strided(_cloud(case["kind"], n, seed)[0], case["stride"]), out=zeros(n, 4),
                  n_out=zeros(1, dtype=torch.int64), assign=zeros(n, dtype=torch.int32) if case["assign"] else False)
    elif op == "ground":
        n = case["n"]
        st.update(xyz=_strided(_cloud("lidar", n, seed)[0], case["stride"]), out=zeros(n, case["stride"]),
                  n_out=zeros(1, dtype=torch.int64), params=kmx.ground_params_default())
    elif op == "features":
        n = case["n"]
        xyz, voxel, vp = _voxel_cloud(case["kind"], n, seed)
        points = _strided(xyz, 4)
        params = kmx.params_default(voxel, viewpoint=np.float32(vp).tolist())
        out = dict(normal4=zeros(n, 4), flags=zeros(n, dtype=torch.uint8), desc=zeros(n, kmx.DESC_STRIDE),
                   valid=zeros(n, dtype=torch.int32), n_valid=zeros(1, dtype=torch.int64))
        if case["method"] == "lists":
            cap = n * {"cube": 256, "lidar": 128, "room": 256}[case["kind"]]  # room for the lists
            out.update(offs=zeros(n + 1, dtype=torch.int64), nbr=zeros(cap, dtype=torch.int32),
                       needed=zeros(1, dtype=torch.int64))
        st.update(points=points, params=params, out=out, grid=ctx.build_grid(points, params.r_fpfh))
    elif op == "match":
        cap = min(case["n_src"], case["n_tgt"])
        st.update(src=_rows(case["kind"], case["n_src"], seed, 0), tgt=_rows(case["kind"], case["n_tgt"], seed, 1),
                  ids=[torch.arange(case[k], dtype=torch.int32, device=DEV) for k in ("n_src", "n_tgt")],
                  corr=zeros(cap, 4, dtype=torch.int32), n_corr=zeros(1, dtype=torch.int64),
                  mode=kmx.MATCH_FP32_EXACT if case["mode"] == "fp32" else kmx.MATCH_BF16_RERANK)
    elif op == "register":
        corr, a, b, beta = _register_problem(case, seed)
        k = case["n_tau"]
        i32 = torch.int32
        st.update(corr=corr, a=a, b=b, beta=beta,
                  pruned=dict(sel=zeros(k, dtype=i32), n_sel=zeros(1, dtype=torch.int64), core=zeros(k, dtype=i32),
                              kmax=zeros(1, dtype=i32), inlier=zeros(k, dtype=i32), n_inlier=zeros(1, dtype=torch.int64)),
                  pose=dict(R=zeros(9, dtype=F64), t=zeros(3, dtype=F64), w=zeros(k), stats=zeros(4, dtype=i32)))
    else:
        ns, nt = case["n_src"], case["n_tgt"]
        pair = pipeline.PairState(ctx, ns, nt)
        params = []
        for side, n, view in ((pair.src, ns, 0), (pair.tgt, nt, 1)):
            xyz, vp = _cloud(case["kind"], n, seed, view)
            side.raw.copy_(xyz)
            params.append(kmx.params_default(case["voxel"], viewpoint=np.float32(vp).tolist()))
            for t in (side.vox4, side.bufs["normal4"], side.bufs["flags"], side.out["desc"], side.out["valid"]):
                t.zero_()
            if case["suppress"]:
                side.suppress = kmx.ground_params_default()
        pair.corr.zero_()
        mode = kmx.MATCH_FP32_EXACT if case["mode"] == "fp32" else kmx.MATCH_BF16_RERANK
        torch.cuda.synchronize()
        pair.run_checked(ns, nt, *params, mode)
        st.update(pair=pair, graph=pair.capture(ns, nt, *params, mode))
    return st


def _corr_out(kmx, corr, n):
    i, j, d1, d2 = kmx.corr_fields(corr, corr.shape[0])
    return dict(i=i, j=j, d1=d1, d2=d2, n=n)


def run(state):
    from paper_2409_15615_gb300 import kmx

    ctx, op, case = state["ctx"], state["op"], state["case"]
    if op == "voxelize":
        out, n, assign = ctx.voxelize(state["xyz"], case["voxel"], out4=state["out"], n_out=state["n_out"],
                                      assign=state["assign"])
        return dict(out=out, n=n) if assign is None else dict(out=out, n=n, assign=assign)
    if op == "ground":
        r = ctx.suppress_ground(state["xyz"], state["params"], out=state["out"], n_out=state["n_out"])
        return dict(out=r["out"], n=r["n_out"])
    if op == "features":
        prm, out = state["params"], state["out"]
        grid = ctx.build_grid(state["points"], prm.r_fpfh, reuse=state["grid"])
        if case["method"] == "faster":
            r = ctx.features(grid, prm, out=out)
            return {k: r[k] for k in ("normal4", "flags", "desc", "valid", "n_valid")}
        a = ctx.normals(grid, prm, out["nbr"].numel(), out=out)
        b = ctx.fasterpfh(grid, prm, a["normal4"], a["flags"], a["offs"], a["nbr"], out=out)
        return dict(normal4=a["normal4"], flags=a["flags"], offs=a["offs"], nbr=a["nbr"], needed=a["needed"],
                    desc=b["desc"], valid=b["valid"], n_valid=b["n_valid"])
    if op == "match":
        corr, n = ctx.match(state["src"], state["ids"][0], case["n_src"], state["tgt"], state["ids"][1], case["n_tgt"],
                            mode=state["mode"], out=state["corr"], n_out=state["n_corr"])
        return _corr_out(kmx, corr, n)
    if op == "register":
        pr = ctx.prune(state["corr"], state["corr"].shape[0], state["a"], state["b"], state["beta"],
                       n_tau=case["n_tau"], out=state["pruned"])
        pose = ctx.gnc(state["corr"], pr, state["a"], state["b"], state["beta"], out=state["pose"])
        return dict(pr, **pose)
    state["graph"].replay()
    pair = state["pair"]
    out = _corr_out(kmx, pair.corr, pair.n_corr)
    for name, c in (("src", pair.src), ("tgt", pair.tgt)):
        out[name] = dict(vox=c.vox4, n_vox=c.n_vox, desc=c.out["desc"], valid=c.out["valid"],
                         n_valid=c.out["n_valid"], normal4=c.bufs["normal4"], flags=c.bufs["flags"])
    return out


# ---------------------------------------------------------------------------
# the results in 64 bits
# ---------------------------------------------------------------------------

def _padded(x, rows, cols=None):
    """x in the first rows of a zero array of the output's shape, FP64."""
    out = torch.zeros((rows,) if cols is None else (rows, cols), dtype=F64, device=DEV)
    if cols is None:
        out[:len(x)] = x
    else:
        out[:len(x), :x.shape[1]] = x
    return out


def _core_numbers64(adj):
    """Core numbers of a dense boolean graph by peeling."""
    left = torch.ones(len(adj), dtype=torch.bool, device=DEV)
    a = adj.float()
    core = torch.zeros(len(adj), dtype=torch.long, device=DEV)
    k = 0
    while bool(left.any()):
        deg = torch.where(left, a @ left.float(), float("inf"))
        k = max(k, int(deg.min()))
        gone = deg <= k
        core[gone] = k
        left &= ~gone
    return core


def _fit64(a, b, w):
    ca, cb = (w[:, None] * a).sum(0) / w.sum(), (w[:, None] * b).sum(0) / w.sum()
    u, _, vt = np.linalg.svd(((a - ca) * w[:, None]).T @ (b - cb))
    R = vt.T @ np.diag([1, 1, np.sign(np.linalg.det(vt.T @ u.T))]) @ u.T
    return R, cb - R @ ca


def _gnc64(a, b, c):
    """GNC with the truncated-least-squares loss around the weighted rigid fit."""
    w, c2 = np.ones(len(a)), c * c
    R, t = _fit64(a, b, w)
    r2 = ((b - a @ R.T - t) ** 2).sum(1)
    if r2.max() <= c2:
        return R, t, w
    mu, last = c2 / max(2 * r2.max() - c2, 1e-30), np.inf
    for _ in range(100):
        lo, hi = mu / (mu + 1) * c2, (mu + 1) / mu * c2
        w = np.where(r2 <= lo, 1.0, np.where(r2 >= hi, 0.0, c * math.sqrt(mu * (mu + 1)) / np.sqrt(np.maximum(r2, 1e-300)) - mu))
        if np.count_nonzero(w > 0) < 3:
            break
        R, t = _fit64(a, b, w)
        r2 = ((b - a @ R.T - t) ** 2).sum(1)
        cost = float((w * r2).sum())
        if abs(cost - last) < 1e-12:
            break
        last, mu = cost, 1.4 * mu
    return R, t, w


def exact(case, seed):
    op = case["op"]
    if op == "voxelize":
        n = case["n"]
        xyz = _cloud(case["kind"], n, seed)[0]
        out = dict(out=_padded(_voxels64(xyz, case["voxel"]), n, 4), n=None)
        return dict(out, assign=None) if case["assign"] else out
    if op == "features":
        n = case["n"]
        normal4, _, desc = _descriptors64(*_voxel_cloud(case["kind"], n, seed))
        out = dict(normal4=normal4, flags=None, desc=_padded(desc, n, 36), valid=None, n_valid=None)
        return dict(out, offs=None, nbr=None, needed=None) if case["method"] == "lists" else out
    if op == "match":
        ns, nt = case["n_src"], case["n_tgt"]
        if ns * nt > EXACT_PAIRS:
            return None
        x, y = _rows(case["kind"], ns, seed, 0)[:, :33].double(), _rows(case["kind"], nt, seed, 1)[:, :33].double()
        near, d1, d2, back = _nearest64(x, y)
        keep = back[near] == torch.arange(ns, device=DEV)
        cap = min(ns, nt)
        return dict(i=None, j=None, d1=_padded(d1[keep], cap), d2=_padded(d2[keep], cap), n=None)
    if op == "register":
        corr, a4, b4, beta = _register_problem(case, seed)
        ratio = corr[:, 2].view(torch.float32).double() / corr[:, 3].view(torch.float32).double()
        sel = torch.argsort(ratio, stable=True)[:case["n_tau"]]
        a, b = a4[corr[sel, 0].long(), :3].double(), b4[corr[sel, 1].long(), :3].double()
        far = lambda p: torch.sqrt(((p[:, None] - p[None]) ** 2).sum(2))  # noqa: E731
        adj = (far(b) - far(a)).abs() <= 2 * beta
        adj.fill_diagonal_(False)
        core = _core_numbers64(adj)
        keep = core == core.max()
        R, t, w = _gnc64(a[keep].cpu().numpy(), b[keep].cpu().numpy(), beta)
        return dict(sel=None, n_sel=None, core=None, kmax=None, inlier=None, n_inlier=None, R=R.reshape(9), t=t,
                    w=_padded(torch.tensor(w, device=DEV), case["n_tau"]), stats=None)
    if op == "pair":
        if case["suppress"]:
            return None
        out = dict(i=None, j=None, d1=None, d2=None, n=None)
        for name, n, view in (("src", case["n_src"], 0), ("tgt", case["n_tgt"], 1)):
            xyz, vp = _cloud(case["kind"], n, seed, view)
            vox = _voxels64(xyz, case["voxel"])
            normal4, _, desc = _descriptors64(vox.float(), case["voxel"], vp)
            out[name] = dict(vox=_padded(vox, n, 4), n_vox=None, desc=_padded(desc, n, 36), valid=None, n_valid=None,
                             normal4=_padded(normal4, n, 4), flags=None)
        return out
    return None  # ground suppression copies the points that it keeps: nothing is rounded
