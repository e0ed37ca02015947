"""Performance cases of the VGICP library: what a mapping program has it do.

A LiDAR mapping program (arXiv 2202.00242) preprocesses each scan (voxel-grid
downsampling, k-NN covariances), registers it against the keyframes of a sliding
window (map rebuild and a handful of factors, or one factor in a Gauss-Newton
loop), and optimizes a global map (hundreds of submaps, thousands of factors
re-linearized together), with overlap rates deciding which factors exist.  Each
kind of case below is one of these calls, made through ``api`` / ``autograd``.

Inputs are synthetic scenes drawn on the GPU from the seed: a room, a corridor
window, and submaps along two laps of a city loop, with the sizes, noise levels
and pose errors of the repository's own workloads.  Point covariances are
I - (1 - 1e-3) n n^T for the surface normal n, the structure the k-NN estimate
has after regularisation.

    listed()             the measured cases
    draw(rng)            another case of the same ranges
    prepare(case, seed)  inputs, maps and plans a program holds before the call
    run(state)           one pass; its outputs
    work(case)           bytes and operations the pass cannot do without
    exact(case, seed)    the outputs in binary64, from plain torch
"""
import math

import numpy as np
import torch

from paper_2202_00242_gb300 import api, autograd

EPS = 1e-3          # regularised small eigenvalue
SPLIT = 0.01        # time split of a 0.1 s sweep (s)
FLOP_TERM = 211.0   # one point-voxel term (H, b, err)
FLOP_POINT = 29.0   # transform and key of a source point


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # one factor of 8,192 points in a room: a Gauss-Newton iteration of the
        # front end, the smallest call a program repeats
        {"name": "factor", "kind": "factor", "n": 8192, "resolution": 0.5, "neighbours": 1},
        # the same factor with 27-neighbour correspondences (coarse alignment)
        {"name": "factor_27", "kind": "factor", "n": 8192, "resolution": 0.5, "neighbours": 27},
        # point covariances of one incoming scan
        {"name": "scan_covariances", "kind": "covariances", "clouds": 1, "n_min": 20000,
         "n_max": 20000, "k": 10, "lists": False},
        # point covariances of a batch of submaps (a map loaded without them)
        {"name": "submap_covariances", "kind": "covariances", "clouds": 64, "n_min": 30000,
         "n_max": 80000, "k": 10, "lists": False},
        # voxel-grid downsampling of one raw sweep with its timestamps
        {"name": "scan_downsample", "kind": "downsample", "clouds": 1, "n": 60000,
         "resolution": 0.25, "split": True},
        # one front-end window: 10 keyframe maps rebuilt, 10 factors of the latest
        # scan linearized, at the fine and at the coarse voxel size
        {"name": "window_fine", "kind": "window", "keyframes": 10, "n": 20000,
         "resolution": 0.25},
        {"name": "window_coarse", "kind": "window", "keyframes": 10, "n": 20000,
         "resolution": 1.0},
        # the global map: 500 submaps rebuilt, 5,000 factors linearized
        {"name": "global_step", "kind": "global", "submaps": 500, "n_min": 30000,
         "n_max": 80000, "per_source": 10, "resolution": 1.0, "rebuild": True,
         "sources": "maps"},
        # re-linearization at new poses only, sources in the order they were captured
        {"name": "relinearize_clouds", "kind": "global", "submaps": 100, "n_min": 30000,
         "n_max": 80000, "per_source": 10, "resolution": 1.0, "rebuild": False,
         "sources": "clouds"},
        # differentiable costs of 256 factors: forward and backward over se(3)
        {"name": "differentiable", "kind": "differentiable", "submaps": 64, "n_min": 20000,
         "n_max": 50000, "per_source": 4, "resolution": 1.0, "exact": False},
        # overlap rates of every ordered pair of 60 submaps (factor creation)
        {"name": "overlap", "kind": "overlap", "submaps": 60, "n_min": 30000, "n_max": 80000,
         "resolution": 1.0},
        # dense 27-neighbour linearization of one resident batch of a large map
        {"name": "dense_27", "kind": "dense", "submaps": 48, "n_min": 100000, "n_max": 100000,
         "per_source": 20, "resolution": 0.5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["factor", "factor", "covariances", "covariances", "downsample", "window",
                       "window", "global", "global", "differentiable", "overlap", "dense"])
    if kind == "factor":
        return {"kind": kind, "n": _log_int(rng, 1000, 60000),
                "resolution": rng.choice([0.25, 0.5, 1.0]), "neighbours": rng.choice([1, 27])}
    if kind == "covariances":
        hi = _log_int(rng, 3000, 80000)
        return {"kind": kind, "clouds": _log_int(rng, 1, 24), "n_min": max(500, hi // 3),
                "n_max": hi, "k": rng.choice([5, 10, 10, 20]), "lists": rng.random() < 0.25}
    if kind == "downsample":
        return {"kind": kind, "clouds": rng.choice([1, 1, 4]), "n": _log_int(rng, 4000, 250000),
                "resolution": rng.choice([0.1, 0.25, 0.5, 1.0]), "split": rng.random() < 0.7}
    if kind == "window":
        return {"kind": kind, "keyframes": rng.randint(2, 20), "n": _log_int(rng, 2000, 40000),
                "resolution": rng.choice([0.25, 0.5, 1.0])}
    if kind == "global":
        hi = _log_int(rng, 20000, 80000)
        return {"kind": kind, "submaps": _log_int(rng, 12, 200), "n_min": hi * 3 // 8,
                "n_max": hi, "per_source": rng.randint(4, 10),
                "resolution": rng.choice([0.5, 1.0, 1.0]), "rebuild": rng.random() < 0.5,
                "sources": rng.choice(["maps", "clouds"])}
    if kind == "differentiable":
        hi = _log_int(rng, 5000, 50000)
        return {"kind": kind, "submaps": _log_int(rng, 8, 64), "n_min": hi * 2 // 5, "n_max": hi,
                "per_source": rng.randint(2, 4), "resolution": rng.choice([0.5, 1.0]),
                "exact": rng.random() < 0.5}
    if kind == "overlap":
        hi = _log_int(rng, 10000, 80000)
        return {"kind": kind, "submaps": _log_int(rng, 6, 60), "n_min": hi * 3 // 8, "n_max": hi,
                "resolution": rng.choice([0.5, 1.0])}
    hi = _log_int(rng, 20000, 100000)
    return {"kind": kind, "submaps": rng.randint(6, 32), "n_min": hi, "n_max": hi,
            "per_source": rng.randint(3, 5) if hi < 50000 else rng.randint(2, 5),
            "resolution": 0.5}


# ---------------------------------------------------------------------------
# scenes, drawn on the GPU
# ---------------------------------------------------------------------------

def _rot(axis, angle):
    a = np.asarray(axis, float) / np.linalg.norm(axis)
    K = np.array([[0, -a[2], a[1]], [a[2], 0, -a[0]], [-a[1], a[0], 0]])
    return np.eye(3) + math.sin(angle) * K + (1 - math.cos(angle)) * (K @ K)


def _pose(R, t):
    T = np.eye(4)
    T[:3, :3], T[:3, 3] = R, t
    return T


def _perturbed(rng, T, sigma_t, sigma_deg):
    w = np.radians(sigma_deg) * rng.normal(size=3)
    return T @ _pose(_rot(w, np.linalg.norm(w)), sigma_t * rng.normal(size=3))


def _random(seed):
    """A host and a device generator of their own for each seed."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (seed + 1) % (2 ** 62))
    return np.random.default_rng(seed), g


def _uniform(g, *shape):
    return torch.rand(*shape, dtype=torch.float64, device="cuda", generator=g)


def _normal(g, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=g)


def _covs(n):
    s = 1.0 - EPS
    return torch.stack([1.0 - s * n[:, 0] * n[:, 0], -s * n[:, 0] * n[:, 1],
                        -s * n[:, 0] * n[:, 2], 1.0 - s * n[:, 1] * n[:, 1],
                        -s * n[:, 1] * n[:, 2], 1.0 - s * n[:, 2] * n[:, 2]],
                       1).float().contiguous()


def _box(g, n, size, origin, sigma):
    """Points uniform by area on the six faces of a box, and their normals."""
    L = torch.tensor(size, dtype=torch.float64, device="cuda")
    area = torch.stack([L[1] * L[2], L[0] * L[2], L[0] * L[1]]).repeat_interleave(2)
    face = torch.multinomial(area, n, replacement=True, generator=g)
    axis, side = face // 2, (face % 2).double()
    u = _uniform(g, n, 3) * L
    u.scatter_(1, axis[:, None], (side * L[axis])[:, None])
    nrm = torch.zeros(n, 3, dtype=torch.float64, device="cuda")
    nrm.scatter_(1, axis[:, None], (1.0 - 2.0 * side)[:, None])
    return u + torch.tensor(origin, dtype=torch.float64, device="cuda") + sigma * _normal(g, n, 3), nrm


def _into(T, p, n):
    """World points and normals in the frame whose world pose is T."""
    R = torch.tensor(T[:3, :3], dtype=torch.float64, device="cuda")
    t = torch.tensor(T[:3, 3], dtype=torch.float64, device="cuda")
    return (p - t) @ R, n @ R


def _room(case, seed):
    """Target and source of a 10 x 10 x 3 m room, the source displaced by 5 deg and 0.2 m."""
    rng, g = _random(seed)
    origin = np.array([-5.0, -5.0, -1.5]) + rng.uniform(-0.2, 0.2, 3)
    out = []
    T = _pose(_rot(rng.normal(size=3), math.radians(5.0)), 0.2 * _unit(rng))
    for pose in (np.eye(4), T):
        p, n = _box(g, case["n"], (10.0, 10.0, 3.0), origin, 0.01)
        p, n = _into(pose, p, n)
        out.append((p.float().contiguous(), _covs(n)))
    # a pose on the way to the optimum
    return out[0], out[1], _perturbed(rng, T, 0.05, 1.0)


def _unit(rng):
    v = rng.normal(size=3)
    return v / np.linalg.norm(v)


def _corridor(case, seed):
    """A scan and the keyframes before it, 0.5 m and 3 deg apart, in a corridor of
    floor, ceiling, walls and random pillars; clouds 0..K-1 are the keyframes."""
    rng, g = _random(seed)
    K, n, sigma, half, height = case["keyframes"], case["n"], 0.02, 2.5, 3.0
    pillars = torch.tensor(np.column_stack([rng.uniform(-20, 40, 40), rng.uniform(-1.8, 1.8, 40),
                                            rng.uniform(0.1, 0.3, 40)]), device="cuda")
    clouds, world, R = [], [], np.eye(3)
    for i in range(K + 1):
        if i:
            R = R @ _rot(rng.normal(size=3), math.radians(3.0))
        T = _pose(R, np.array([0.5 * i, 0.0, 1.2]))
        world.append(T)
        what = _uniform(g, n)
        x = T[0, 3] + 40.0 * (_uniform(g, n) - 0.5)
        v, side = _uniform(g, n), (_uniform(g, n) < 0.5).double() * 2.0 - 1.0
        flat = what < 0.3                      # floor (60 %) or ceiling
        top = (_uniform(g, n) < 0.4).double()
        c = pillars[torch.randint(0, 40, (n,), device="cuda", generator=g)]
        th = 2.0 * math.pi * _uniform(g, n)
        post = what > 0.86
        p = torch.stack([x, side * half, height * v], 1)
        nrm = torch.stack([torch.zeros_like(x), -side, torch.zeros_like(x)], 1)
        p = torch.where(flat[:, None], torch.stack([x, half * (2 * v - 1), height * top], 1), p)
        nrm = torch.where(flat[:, None],
                          torch.stack([0 * x, 0 * x, 1.0 - 2.0 * top], 1), nrm)
        p = torch.where(post[:, None], torch.stack([c[:, 0] + c[:, 2] * th.cos(),
                                                    c[:, 1] + c[:, 2] * th.sin(),
                                                    height * v], 1), p)
        nrm = torch.where(post[:, None], torch.stack([th.cos(), th.sin(), 0 * x], 1), nrm)
        p, nrm = _into(T, p + sigma * _normal(g, n, 3), nrm)
        clouds.append((p.float().contiguous(), _covs(nrm)))
    pairs = np.array([[k, K] for k in range(K)], np.int32)
    poses = np.stack([_perturbed(rng, np.linalg.inv(world[k]) @ world[K], 0.02, 0.3)
                      for k in range(K)])
    return clouds, pairs, poses


def _sizes(case, rng):
    """Point counts spread log-uniformly over [n_min, n_max], in random order."""
    C = case.get("submaps") or case["clouds"]
    lo, hi = case["n_min"], case["n_max"]
    s = np.exp(math.log(lo) + (np.arange(C) + 0.5) / C * (math.log(hi) - math.log(lo)))
    return rng.permutation(s.astype(np.int64))


def _city(sizes, spacing, rng, g, sigma=0.03, radius=40.0):
    """Submaps along two laps of a city loop with box buildings on both sides, each
    in its own frame, points in random order.  Returns (points, covs, offsets,
    world poses, centres)."""
    C = len(sizes)
    a = max(C * spacing / 2.0, 150.0) / 6.0
    knots = np.array([0.0, 2 * a, 3 * a, 5 * a, 6 * a])

    def path(u):
        u = np.mod(u, 6 * a)
        x = np.interp(u, knots, [-a, a, a, -a, -a])
        y = np.interp(u, knots, [-a / 2, -a / 2, a / 2, a / 2, -a / 2])
        h = np.array([0.0, 0.5, 1.0, 1.5])[np.clip(np.searchsorted(knots, u, "right") - 1, 0, 3)]
        return x, y, h * math.pi

    u = np.arange(C) * (12 * a / C)
    x, y, h = path(u)
    lap = np.floor(u / (6 * a))
    x, y = x - 3.0 * lap * np.sign(x), y - 3.0 * lap * np.sign(y)
    seg, zs = [], []
    for bx, by, bh in zip(*path(np.arange(0.0, 6 * a, 20.0))):
        for side in (-1.0, 1.0):
            if rng.random() < 0.15:
                continue
            off, w, d, top = rng.uniform(12, 20), rng.uniform(8, 18), rng.uniform(8, 18), rng.uniform(6, 30)
            c = np.array([bx, by]) + side * off * np.array([-math.sin(bh), math.cos(bh)])
            ex, ey = np.array([math.cos(bh), math.sin(bh)]), np.array([-math.sin(bh), math.cos(bh)])
            q = [c + i * w / 2 * ex + j * d / 2 * ey for i, j in ((-1, -1), (1, -1), (1, 1), (-1, 1))]
            for k in range(4):
                seg.append(np.r_[q[k], q[(k + 1) % 4]])
                zs.append(top)
    seg, zs = np.array(seg), np.array(zs)
    length = np.hypot(seg[:, 2] - seg[:, 0], seg[:, 3] - seg[:, 1])
    centre = np.column_stack([x, y])
    mid = 0.5 * (seg[:, :2] + seg[:, 2:])
    dist = np.linalg.norm(mid[None] - centre[:, None], axis=2)
    weight = np.where(dist < radius + 5.0, length * np.minimum(zs, radius), 0.0)
    weight[:, 0] += 1e-9
    world = [_pose(_rot([0, 0, 1], h[i] + rng.uniform(-0.2, 0.2)) @
                   _rot(rng.normal(size=3), math.radians(rng.uniform(0.0, 2.0))),
                   np.array([x[i], y[i], 1.8])) for i in range(C)]

    def dev(v):
        return torch.tensor(np.asarray(v), dtype=torch.float64, device="cuda")

    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pts = torch.empty(int(off[-1]), 3, dtype=torch.float32, device="cuda")
    cov = torch.empty(int(off[-1]), 6, dtype=torch.float32, device="cuda")
    seg_d, z_d, w_d, c_d = dev(seg), dev(zs), dev(weight), dev(np.column_stack([x, y, 0 * x + 1.8]))
    R_d, t_d = dev([T[:3, :3] for T in world]), dev([T[:3, 3] for T in world])
    for i0 in range(0, C, 64):  # 64 submaps at a time
        i1 = min(C, i0 + 64)
        m = int(max(sizes[i0:i1]))
        rows = torch.arange(m, device="cuda")[None] < torch.tensor(sizes[i0:i1], device="cuda")[:, None]
        pick = torch.multinomial(w_d[i0:i1], m, replacement=True, generator=g)[rows]
        sub = torch.arange(i0, i1, device="cuda")[:, None].expand(-1, m)[rows]
        n = pick.shape[0]
        s, z, ground = _uniform(g, n), _uniform(g, n), _uniform(g, n) < 0.35
        e = seg_d[pick]
        d = e[:, 2:] - e[:, :2]
        p = torch.cat([e[:, :2] + s[:, None] * d, (z * z_d[pick])[:, None]], 1)
        nrm = torch.stack([-d[:, 1], d[:, 0], 0 * s], 1)
        nrm = nrm / nrm.norm(dim=1, keepdim=True)
        ground |= (p - c_d[sub]).norm(dim=1) > radius  # out of range: the ground instead
        r, th = radius * s.sqrt(), 2.0 * math.pi * z
        flat = torch.stack([c_d[sub, 0] + r * th.cos(), c_d[sub, 1] + r * th.sin(), 0 * s], 1)
        up = torch.tensor([0.0, 0.0, 1.0], dtype=torch.float64, device="cuda").expand(n, 3)
        p = torch.where(ground[:, None], flat, p) + sigma * _normal(g, n, 3)
        nrm = torch.where(ground[:, None], up, nrm)
        Rs = R_d[sub]
        pts[off[i0]:off[i1]] = torch.einsum("na,nab->nb", p - t_d[sub], Rs).float()
        cov[off[i0]:off[i1]] = _covs(torch.einsum("na,nab->nb", nrm, Rs))
    return pts, cov, off, world, centre


def _submaps(case, seed, noise):
    """Submaps, the pairs of each with its nearest others, and their perturbed poses."""
    rng, g = _random(seed)
    sizes = _sizes(case, rng)
    spacing = 3.0 if case["kind"] == "dense" else 6.0
    pts, cov, off, world, centre = _city(sizes, spacing, rng, g)
    C = len(sizes)
    if case["kind"] == "overlap":
        pairs = np.array([[j, i] for j in range(C) for i in range(C) if i != j], np.int32)
    else:
        dist = np.linalg.norm(centre[:, None] - centre[None], axis=2)
        np.fill_diagonal(dist, np.inf)
        near = np.argsort(dist, axis=1, kind="stable")[:, :min(case["per_source"], C - 1)]
        pairs = np.array([[j, i] for i in range(C) for j in near[i]], np.int32)
    inv = [np.linalg.inv(T) for T in world]
    poses = np.stack([_perturbed(rng, inv[j] @ world[i], *noise) if noise else inv[j] @ world[i]
                      for j, i in pairs])
    return pts, cov, off, pairs, poses


_NOISE = {"global": (0.1, 1.0), "dense": (0.1, 1.0), "differentiable": (0.3, 5.0), "overlap": None}


def _sweep(case, seed):
    """Raw sweeps of a spinning LiDAR in a street: slightly more than one turn, points in time
    order, each with its timestamp."""
    rng, g = _random(seed)
    pts, times = [], []
    for _ in range(case["clouds"]):
        n = case["n"]
        i = torch.arange(n, dtype=torch.float64, device="cuda") / n
        th = 2.0 * math.pi * 1.08 * i + rng.uniform(0.0, 6.0)
        el = torch.deg2rad(-20.0 + 35.0 * _uniform(g, n))
        # range to the nearest of the ground, two house fronts and a far limit
        far = torch.full_like(i, 60.0)
        front = (9.0 + rng.uniform(0.0, 3.0)) / (th.sin().abs() * el.cos()).clamp_min(1e-3)
        floor = torch.where(el < 0, 1.8 / (-el.sin()).clamp_min(1e-3), far)
        r = torch.minimum(torch.minimum(front, floor), far) * (1.0 + 0.002 * _normal(g, n))
        pts.append(torch.stack([r * th.cos() * el.cos(), r * th.sin() * el.cos(), r * el.sin()], 1))
        times.append(0.1 * i)
    off = np.arange(case["clouds"] + 1, dtype=np.int64) * case["n"]
    return (torch.cat(pts).float().contiguous(),
            torch.cat(times).float().contiguous() if case["split"] else None, off)


def _clouds(case, seed):
    rng, g = _random(seed)
    return _city(_sizes(case, rng), 6.0, rng, g)[:3]


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "factor":
        (tp, tc), (sp, sc), T = _room(case, seed)
        return {"case": case, "map": api.VoxelMap.build(tp, tc, case["resolution"]),
                "src": (sp, sc), "T": T}
    if kind == "covariances":
        pts, _, off = _clouds(case, seed)
        return {"case": case, "points": pts, "offsets": off}
    if kind == "downsample":
        pts, times, off = _sweep(case, seed)
        return {"case": case, "points": pts, "times": times, "offsets": off}
    if kind == "window":
        clouds, pairs, poses = _corridor(case, seed)
        pts = torch.cat([c[0] for c in clouds[:-1]])
        cov = torch.cat([c[1] for c in clouds[:-1]])
        off = np.arange(len(clouds), dtype=np.int64) * case["n"]
        maps = api.build_voxelmaps(pts, cov, off, case["resolution"])
        pairs[:, 1] = 0  # one source: the scan
        plan = api.Plan(maps, [clouds[-1]], pairs)
        return {"case": case, "maps": maps, "clouds": (pts, cov), "plan": plan, "poses": poses,
                "out": _result(len(pairs))}
    pts, cov, off, pairs, poses = _submaps(case, seed, _NOISE[kind])
    maps = api.build_voxelmaps(pts, cov, off, case["resolution"])
    s = {"case": case, "maps": maps, "pairs": pairs, "poses": poses}
    if kind == "global":
        src = maps if case["sources"] == "maps" else [
            (pts[off[c]:off[c + 1]], cov[off[c]:off[c + 1]]) for c in range(len(maps))]
        s |= {"clouds": (pts, cov), "plan": api.Plan(maps, src, pairs), "out": _result(len(pairs))}
    elif kind == "differentiable":
        rng = np.random.default_rng(seed + 7)
        s |= {"factors": autograd.FactorSet(maps, maps, pairs, poses, exact=case["exact"]),
              "xi": torch.tensor(0.01 * rng.normal(size=(len(pairs), 6)), device="cuda",
                                 requires_grad=True),
              "weight": torch.tensor(rng.uniform(0.5, 2.0, len(pairs)), device="cuda")}
    return s


def _result(n_pairs):
    return (torch.empty(n_pairs, api.RESULT_SIZE, dtype=torch.float64, device="cuda"),
            torch.empty(n_pairs, dtype=torch.int64, device="cuda"))


def run(state):
    s, kind = state, state["case"]["kind"]
    if kind == "factor":
        r = api.linearize(s["map"], *s["src"], s["T"], neighbours=s["case"]["neighbours"])
    elif kind == "covariances":
        c = s["case"]
        r = api.estimate_covariances(s["points"], s["offsets"], k=c["k"], neighbours=c["lists"])
        return {"covs": r[0], "lists": r[1]} if c["lists"] else {"covs": r}
    elif kind == "downsample":
        p, t, n, o = api.downsample(s["points"], s["case"]["resolution"], times=s["times"],
                                    split=SPLIT if s["case"]["split"] else 0.0,
                                    offsets=s["offsets"])
        # into scan buffers of a fixed size, as the next stages keep them
        rest = len(s["points"]) - len(p)
        pad = torch.nn.functional.pad
        return {"points": pad(p, (0, 0, 0, rest)), "counts": pad(n, (0, rest)),
                "times": None if t is None else pad(t, (0, rest)), "offsets": o}
    elif kind in ("window", "global"):
        if kind == "window" or s["case"]["rebuild"]:
            api.rebuild_voxelmaps(s["maps"], *s["clouds"])
        r = s["plan"].execute(s["poses"], out=s["out"][0], inliers=s["out"][1])
    elif kind == "differentiable":
        err = s["factors"].cost(s["xi"])
        grad, = torch.autograd.grad((err * s["weight"]).sum(), s["xi"])
        return {"err": err.detach(), "grad": grad}
    elif kind == "overlap":
        rate, n = api.overlap_batched(s["maps"], s["maps"], s["pairs"], s["poses"])
        return {"rate": rate, "inliers": n}
    else:
        r = api.linearize_batched(s["maps"], s["maps"], s["pairs"], s["poses"], neighbours=27)
    return {"result": r.out, "inliers": r.inliers}


def work(case):
    """Every cloud read once (36 B a point; 12 B where covariances are not read), every
    result written once; operations per source point and point-voxel term."""
    kind = case["kind"]
    if kind == "factor":
        near = case["neighbours"]
        n = float(case["n"])
        # the map's voxels (64 B each) as well: at most one a point
        return {"bytes": 36 * n + 64 * min(n, 190.0 / case["resolution"] ** 2) + 352,
                "flops": n * (FLOP_POINT + FLOP_TERM * (1 if near == 1 else 7.3))}
    if kind == "covariances":
        n = float(np.sum(_sizes(case, np.random.default_rng(0))))
        k = case["k"]
        # k candidates' distances, the mean and the scatter of k neighbours, one 3x3 eigenvector
        return {"bytes": n * (12 + 24 + (4 * k if case["lists"] else 0)),
                "flops": n * (k * (8 + 6 + 15) + 300)}
    if kind == "downsample":
        n = float(case["n"] * case["clouds"])
        return {"bytes": n * (12 + (4 if case["split"] else 0)) + 0.3 * n * 20, "flops": n * 20}
    if kind == "window":
        n, K = float(case["n"]), case["keyframes"]
        return {"bytes": 36 * n * (K + 1) + 352 * K,
                "flops": n * K * (FLOP_POINT + FLOP_TERM + 100)}
    s = float(np.sum(_sizes(case, np.random.default_rng(0))))
    C = case["submaps"]
    per = C - 1 if kind == "overlap" else min(case["per_source"], C - 1)
    if kind == "overlap":
        return {"bytes": 12 * s + 8 * C * per, "flops": s * per * FLOP_POINT}
    if kind == "differentiable":
        # cost and gradient of every factor
        return {"bytes": 36 * s + 56 * C * per, "flops": s * per * (2 * FLOP_POINT + 110 + 135)}
    if kind == "dense":
        return {"bytes": 36 * s + 352 * C * per,
                "flops": s * per * (FLOP_POINT + 7.3 * FLOP_TERM)}
    build = 100 if case["rebuild"] else 0  # sums of 9 values, exact
    return {"bytes": 36 * s + 352 * C * per,
            "flops": s * per * (FLOP_POINT + FLOP_TERM) + s * build}


# ---------------------------------------------------------------------------
# the same in binary64
# ---------------------------------------------------------------------------

def _keys(q, r):
    k = torch.floor(q / r).to(torch.int64) + (1 << 20)
    return (k[:, 0] << 42) | (k[:, 1] << 21) | k[:, 2]


def _map64(pts, cov, r):
    """Sorted voxel keys, mean positions and mean covariances (upper triangles)."""
    k, at = torch.unique(_keys(pts.double(), r), return_inverse=True)
    n = torch.zeros(len(k), dtype=torch.float64, device="cuda").index_add_(
        0, at, torch.ones(len(at), dtype=torch.float64, device="cuda"))
    s = torch.zeros(len(k), 9, dtype=torch.float64, device="cuda").index_add_(
        0, at, torch.cat([pts, cov], 1).double())
    s /= n[:, None]
    return k, s[:, :3], s[:, 3:]


_FULL = [0, 1, 2, 1, 3, 4, 2, 4, 5]


def _transformed(p, T):
    return torch.stack([((T[a, 0] * p[:, 0] + T[a, 1] * p[:, 1]) + T[a, 2] * p[:, 2]) + T[a, 3]
                        for a in range(3)], 1)


def _matches(vmap, q, r, offset=None):
    """(rows of q with a voxel, their voxels)."""
    k = torch.floor(q / r).to(torch.int64) + (1 << 20)
    if offset is not None:
        k = k + offset
    key = (k[:, 0] << 42) | (k[:, 1] << 21) | k[:, 2]
    at = torch.searchsorted(vmap[0], key).clamp_max(len(vmap[0]) - 1)
    hit = torch.nonzero(vmap[0][at] == key)[:, 0]
    return hit, at[hit]


def _weights(vcov, scov, R):
    C = scov[:, _FULL].reshape(-1, 3, 3)
    M = vcov[:, _FULL].reshape(-1, 3, 3) + R @ C @ R.T
    a, b, c, d, e, f = (M[:, 0, 0], M[:, 0, 1], M[:, 0, 2], M[:, 1, 1], M[:, 1, 2], M[:, 2, 2])
    adj = torch.stack([d * f - e * e, c * e - b * f, b * e - c * d,
                       a * f - c * c, b * c - a * e, a * d - b * b], 1)
    det = a * adj[:, 0] + b * adj[:, 1] + c * adj[:, 2]
    return (adj / det[:, None])[:, _FULL].reshape(-1, 3, 3)


def _factor64(vmap, pts, cov, T, r, neighbours):
    """H, b, err (43 values) and the term count of one factor."""
    p, c, R = pts.double(), cov.double(), torch.tensor(T[:3, :3], device="cuda")
    q = _transformed(p, T)
    H = torch.zeros(6, 6, dtype=torch.float64, device="cuda")
    b = torch.zeros(6, dtype=torch.float64, device="cuda")
    err = torch.zeros((), dtype=torch.float64, device="cuda")
    count = 0
    shifts = [None] if neighbours == 1 else [
        torch.tensor([x, y, z], device="cuda") for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]
    for o in shifts:
        hit, at = _matches(vmap, q, r, o)
        count += len(hit)
        d = vmap[1][at] - q[hit]
        W = _weights(vmap[2][at], c[hit], R)
        m = p[hit]
        J = torch.zeros(len(hit), 3, 6, dtype=torch.float64, device="cuda")
        S = torch.zeros(len(hit), 3, 3, dtype=torch.float64, device="cuda")
        S[:, 0, 1], S[:, 0, 2], S[:, 1, 2] = -m[:, 2], m[:, 1], -m[:, 0]
        S[:, 1, 0], S[:, 2, 0], S[:, 2, 1] = m[:, 2], -m[:, 1], m[:, 0]
        J[:, :, :3], J[:, :, 3:] = R @ S, -R
        WJ = W @ J
        H += J.reshape(-1, 6).T @ WJ.reshape(-1, 6)
        b += WJ.reshape(-1, 6).T @ d.reshape(-1)
        err += ((W @ d[:, :, None])[:, :, 0] * d).sum()
    return torch.cat([H.reshape(-1), b, err[None]]), count


def _cost64(vmap, pts, cov, T0, xi, r, exact):
    """err and its gradient over xi at T0 Exp(xi), by automatic differentiation."""
    x = xi.clone().requires_grad_(True)
    z = torch.zeros((), dtype=torch.float64, device="cuda")
    A = torch.stack([torch.stack([z, -x[2], x[1], x[3]]), torch.stack([x[2], z, -x[0], x[4]]),
                     torch.stack([-x[1], x[0], z, x[5]]), torch.stack([z, z, z, z])])
    T = torch.tensor(T0, device="cuda") @ torch.linalg.matrix_exp(A)
    p, R = pts.double(), T[:3, :3]
    hit, at = _matches(vmap, _transformed(p, T.detach().cpu().numpy()), r)
    d = vmap[1][at] - (p[hit] @ R.T + T[:3, 3])
    W = _weights(vmap[2][at], cov[hit].double(), R if exact else R.detach())
    err = ((W @ d[:, :, None])[:, :, 0] * d).sum()
    g, = torch.autograd.grad(err, x)
    return err.detach(), g


def _covariances64(pts, off, k):
    out = torch.empty(len(pts), 6, dtype=torch.float64, device="cuda")
    for a, b in zip(off[:-1], off[1:]):
        p = pts[a:b]
        n = len(p)
        for i in range(0, n, 2048):
            q = p[i:i + 2048]
            d2 = (q[:, None, 0] - p[None, :, 0]) ** 2
            d2 += (q[:, None, 1] - p[None, :, 1]) ** 2
            d2 += (q[:, None, 2] - p[None, :, 2]) ** 2
            near = torch.topk(d2, min(k + 6, n), dim=1, largest=False).indices
            P = p[near].double()
            e2 = ((P - q[:, None].double()) ** 2).sum(2)
            best = torch.topk(e2, min(k, n), dim=1, largest=False).indices
            P = torch.gather(P, 1, best[:, :, None].expand(-1, -1, 3))
            E = P - P.mean(1, keepdim=True)
            v = torch.linalg.eigh(E.transpose(1, 2) @ E)[1][:, :, 0]
            s = 1.0 - EPS
            out[a + i:a + i + len(q)] = torch.stack(
                [1 - s * v[:, 0] ** 2, -s * v[:, 0] * v[:, 1], -s * v[:, 0] * v[:, 2],
                 1 - s * v[:, 1] ** 2, -s * v[:, 1] * v[:, 2], 1 - s * v[:, 2] ** 2], 1)
    return out


def _first(group, n_groups):
    i = torch.arange(len(group), device="cuda")
    return torch.full((n_groups,), len(group), device="cuda").scatter_reduce_(0, group, i, "amin")


def _downsample64(pts, times, off, r):
    P, T = [], []
    for a, b in zip(off[:-1], off[1:]):
        p = pts[a:b].double()
        key, at = torch.unique(_keys(p, r), return_inverse=True)
        group = 2 * at
        if times is not None:
            t = times[a:b].double()
            group = group + ((t - t[_first(at, len(key))][at]).abs() > SPLIT).long()
        key, at = torch.unique(group, return_inverse=True)
        order = torch.argsort(_first(at, len(key)))
        n = torch.bincount(at, minlength=len(key)).double()
        v = p if times is None else torch.cat([p, t[:, None]], 1)
        s = torch.zeros(len(key), v.shape[1], dtype=torch.float64, device="cuda").index_add_(0, at, v)
        s = (s / n[:, None])[order]
        P.append(s[:, :3])
        if times is not None:
            T.append(s[:, 3])
    return torch.cat(P), torch.cat(T) if T else None


def exact(case, seed):
    kind = case["kind"]
    if kind == "factor":
        (tp, tc), (sp, sc), T = _room(case, seed)
        v, _ = _factor64(_map64(tp, tc, case["resolution"]), sp, sc, T, case["resolution"],
                         case["neighbours"])
        return {"result": v, "inliers": None}
    if kind == "covariances":
        pts, _, off = _clouds(case, seed)
        if float(np.sum(np.diff(off).astype(float) ** 2)) > 3e10:  # the search takes n^2
            return None
        return {"covs": _covariances64(pts, off, case["k"])} | ({"lists": None} if case["lists"] else {})
    if kind == "downsample":
        pts, times, off = _sweep(case, seed)
        p, t = _downsample64(pts, times, off, case["resolution"])
        rest = len(pts) - len(p)
        return {"points": torch.cat([p, p.new_zeros(rest, 3)]), "counts": None, "offsets": None,
                "times": None if t is None else torch.cat([t, t.new_zeros(rest)])}
    r = case["resolution"]
    if kind == "window":
        clouds, pairs, poses = _corridor(case, seed)
        maps = [_map64(*c, r) for c in clouds[:-1]]
        return {"result": torch.stack([_factor64(maps[j], *clouds[i], T, r, 1)[0]
                                       for (j, i), T in zip(pairs, poses)]), "inliers": None}
    pts, cov, off, pairs, poses = _submaps(case, seed, _NOISE[kind])
    cloud = [(pts[a:b], cov[a:b]) for a, b in zip(off[:-1], off[1:])]
    maps = [_map64(*c, r) for c in cloud]
    if kind == "overlap":
        rate = [len(_matches(maps[j], _transformed(cloud[i][0].double(), T), r)[0]) /
                max(1, len(cloud[i][0])) for (j, i), T in zip(pairs, poses)]
        return {"rate": torch.tensor(rate, dtype=torch.float64, device="cuda"), "inliers": None}
    if kind == "differentiable":
        rng = np.random.default_rng(seed + 7)
        xi = torch.tensor(0.01 * rng.normal(size=(len(pairs), 6)), device="cuda")
        weight = torch.tensor(rng.uniform(0.5, 2.0, len(pairs)), device="cuda")
        e, g = zip(*[_cost64(maps[j], *cloud[i], poses[n], xi[n], r, case["exact"])
                     for n, (j, i) in enumerate(pairs)])
        return {"err": torch.stack(e), "grad": torch.stack(g) * weight[:, None]}
    near = 27 if kind == "dense" else 1
    if float(np.sum(np.diff(off)[pairs[:, 1]])) * near > 1.5e9:
        return None  # over 20 seconds of binary64
    return {"result": torch.stack([_factor64(maps[j], *cloud[i], T, r, near)[0]
                                   for (j, i), T in zip(pairs, poses)]), "inliers": None}
