"""The calls whose time this library is judged by, as a user's program makes them.

The work: two scans of a spinning multi-beam scanner over an urban scene (ground, buildings,
cars, poles), scan A registered as a grid's reference, scan B scored under candidate poses.
Sizes are those of the repository's own workloads (8k-point toy scene, 64-beam 120k-point
LiDAR pair on grids of 0.25 to 1 m, 128-beam 260k-point pair on a 6.4M-voxel grid, mixed
batches, served requests, Nelder-Mead restarts); `draw` spreads over the same ranges.

Scans are ray-cast on the GPU (as the synthetic generator of the benchmark does on the host,
but in milliseconds), so that many preparations are cheap.
"""
import math

import numpy as np
import torch

from paper_1709_06948_gb300 import align

COUNT, ZVAR, JOINT = 0, 1, 2
SENSOR = 1.8       # sensor height above the scan frame's origin, m
Z_LOW = -1.0       # grids start 1 m below the ground


# ---------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------
def _case(kind, **kw):
    c = dict(kind=kind, beams=64, az_deg=0.17, points=0, x=160, y=160, z=16, res_mm=500, feature=ZVAR,
             counts="8x8x2x2x2x8", order="345012", half_xy=2.0, half_yaw=5.0, poses=0, levels=0, n=0, iters=0)
    c.update(kw)
    return c


def listed():
    fine = dict(x=320, y=320, z=32, res_mm=250)
    metre = dict(x=80, y=80, z=8, res_mm=1000)
    large = dict(beams=128, az_deg=0.15, x=400, y=400, z=40, res_mm=200, feature=JOINT, half_xy=10.0, half_yaw=30.0)
    return [
        # one candidate pose of an optimiser that runs outside the library: a latency-bound call
        _case("poses", name="one_pose_120k", poses=1),
        # a small scan from host memory against a coarse count grid: the quick check of a toy scene
        _case("lattice_host", name="toy_8k_729_count", points=8000, x=40, y=40, z=8, res_mm=1000, feature=COUNT,
              counts="3x3x3x3x3x3", order="012345", half_xy=1.0),
        # a scan pair aligned from scratch: reference built, six-level lattice search of 4,096 poses each
        _case("search", name="search_120k_6x4096", levels=6),
        # one lattice of candidates on a fine grid (over 20,000 occupied voxels), translations slowest
        _case("lattice", name="lattice_120k_4096_025m", order="012345", **fine),
        # a dense scanner on a coarse grid: voxels of thousands of points
        _case("lattice", name="lattice_260k_dense_1m", beams=128, az_deg=0.15, **metre),
        # scattered candidates on the device (a sampler's or a particle filter's), no two alike
        _case("poses_device", name="scattered_120k_1001", poses=1001),
        # the wide first lattice of the 6.4M-voxel grid with the joint feature: the largest call
        _case("lattice", name="lattice_260k_32768_joint", **dict(large, counts="16x16x2x2x2x16")),
        # that grid's reference built for a new scan A
        _case("reference", name="reference_260k_joint", **large),
        # many pairs of uneven sizes and resolutions in one call, the launch sequence replayed as a graph
        _case("batch", name="batch_12_mixed", n=12),
        # refinement of several candidates by Nelder-Mead in lockstep
        _case("refine", name="refine_120k_16x25", n=16, iters=25),
        # alignment requests served against resident references of four resolutions
        _case("serve", name="serve_12_requests", n=12, levels=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _product(counts):
    p = 1
    for m in counts:
        p *= m
    return p


def draw(rng):
    kind = rng.choice(["poses", "lattice_host", "lattice", "lattice", "lattice", "search", "search", "poses_device",
                       "reference", "batch", "refine", "serve"])
    beams = rng.choice([64, 64, 128])
    res_mm = rng.choice([200, 250, 300, 500, 500, 640, 750, 1000])
    # grids cover 50 to 90 m and 6 to 9 m of height, rarely a round number of voxels
    x, y = (int(rng.uniform(50.0, 90.0) * 1000 / res_mm) for _ in range(2))
    z = max(4, int(rng.uniform(6.0, 9.0) * 1000 / res_mm))
    points = _log_int(rng, 5000, 120000) if rng.random() < 0.6 else 0
    c = _case(kind, beams=beams, az_deg=0.17 if beams == 64 else 0.15, points=points, x=x, y=y, z=z, res_mm=res_mm,
              feature=rng.choice([COUNT, ZVAR, ZVAR, JOINT]), half_xy=round(rng.uniform(0.2, 8.0), 3),
              half_yaw=round(rng.uniform(0.5, 20.0), 3))
    counts = [rng.randint(3, 16), rng.randint(3, 16), rng.randint(1, 3), rng.randint(1, 3), rng.randint(1, 3),
              rng.randint(1, 12)]
    cap = 8192 if kind != "search" else 4096
    while _product(counts) > cap:
        a = rng.randrange(6)
        counts[a] = max(1, counts[a] - 1)
    c["counts"] = "x".join(str(m) for m in counts)
    c["order"] = rng.choice(["345012", "345012", "012345", "201345"])  # rotations or translations slowest
    if kind == "poses":
        c["poses"] = _log_int(rng, 1, 64)
    elif kind == "poses_device":
        c["poses"] = _log_int(rng, 30, 2000)
    elif kind == "search":
        c["levels"] = rng.randint(1, 6)
    elif kind == "batch":
        c["n"] = rng.randint(2, 12)
    elif kind == "refine":
        c["n"], c["iters"] = _log_int(rng, 1, 64), rng.randint(5, 30)
    elif kind == "serve":
        c["n"], c["levels"] = rng.randint(3, 12), rng.randint(2, 6)
    return c


# ---------------------------------------------------------------------------------------
# scans
# ---------------------------------------------------------------------------------------
def _scene(rng):
    """Boxes (buildings along two crossing streets, cars in their lanes) and poles on the kerbs."""
    half = rng.uniform(5.0, 7.0)
    boxes = []

    def place(n, make, gap):
        kept = []
        for _ in range(2000):
            if len(kept) == n:
                break
            b = make()
            if b is not None and all(b[3] + gap < o[0] or o[3] + gap < b[0] or b[4] + gap < o[1] or o[4] + gap < b[1]
                                     for o in kept):
                kept.append(b)
        boxes.extend(kept)

    def building():
        along, depth, length = rng.uniform(-110, 110), rng.uniform(8, 20), rng.uniform(10, 30)
        back, side, height = rng.uniform(8, 15), rng.choice([-1.0, 1.0]), rng.uniform(8, 25)
        lo, hi = (back, back + depth) if side > 0 else (-back - depth, -back)
        if along - length / 2 < half and along + length / 2 > -half:
            return None  # the crossing street stays clear
        b = (along - length / 2, lo, 0.0, along + length / 2, hi, height)
        return b if rng.uniform() < 0.5 else (b[1], b[0], 0.0, b[4], b[3], height)

    def car():
        along, lane = rng.uniform(-60, 60), rng.uniform(-half + 1, half - 1)
        if abs(along) < 6.0:
            return None
        b = (along - 2.25, lane - 0.9, 0.0, along + 2.25, lane + 0.9, 1.5)
        return b if rng.uniform() < 0.5 else (b[1], b[0], 0.0, b[4], b[3], 1.5)

    place(32, building, 1.0)
    place(30, car, 0.5)
    poles = []
    for _ in range(40):
        a, s = rng.uniform(-80, 80), rng.choice([-1.0, 1.0]) * (half + 0.5)
        poles.append((a, s, 0.15, rng.uniform(6, 8)) if rng.uniform() < 0.5 else (s, a, 0.15, rng.uniform(6, 8)))
    return np.array(boxes), np.array(poles)


def _rotation(eta):
    cx, cy, cz = np.cos(eta[3:6])
    sx, sy, sz = np.sin(eta[3:6])
    return (np.array([[cz, -sz, 0], [sz, cz, 0], [0, 0, 1]]) @ np.array([[cy, 0, sy], [0, 1, 0], [-sy, 0, cy]]) @
            np.array([[1, 0, 0], [0, cx, -sx], [0, sx, cx]]))


def _scan(scene, T, beams, az_deg, gen):
    """Returns of a scanner at pose T in its own frame (ring-major, range noise, a tenth of them
    lost), float32 on the GPU."""
    dev, f64 = "cuda", torch.float64
    n_az = int(round(360.0 / az_deg))
    lo, hi, reach = (-24.8, 2.0, 100.0) if beams == 64 else (-25.0, 15.0, 120.0)
    el = torch.deg2rad(torch.linspace(lo, hi, beams, dtype=f64, device=dev))[:, None]
    az = (torch.arange(n_az, dtype=f64, device=dev) * (2 * math.pi / n_az))[None, :]
    d = torch.stack([el.cos() * az.cos(), el.cos() * az.sin(), el.sin().expand(beams, n_az)], -1).reshape(-1, 3)
    R = torch.tensor(_rotation(T), dtype=f64, device=dev)
    t = torch.tensor(T[:3], dtype=f64, device=dev)
    o = R @ torch.tensor([0.0, 0.0, SENSOR], dtype=f64, device=dev) + t
    d = d @ R.T
    d = torch.where(d.abs() < 1e-12, torch.full_like(d, 1e-12), d)
    best = torch.where(d[:, 2] < 0, -o[2] / d[:, 2], math.inf)
    boxes, poles = (torch.tensor(a, dtype=f64, device=dev) for a in scene)
    t1, t2 = (boxes[:, None, :3] - o) / d, (boxes[:, None, 3:] - o) / d
    near, far = torch.minimum(t1, t2).amax(-1), torch.maximum(t1, t2).amin(-1)
    best = torch.minimum(best, torch.where((near <= far) & (near > 1e-6), near, math.inf).amin(0))
    ox, oy = (o[0] - poles[:, 0])[:, None], (o[1] - poles[:, 1])[:, None]
    a, b = d[:, 0] ** 2 + d[:, 1] ** 2, 2 * (ox * d[:, 0] + oy * d[:, 1])
    disc = b * b - 4 * a * (ox * ox + oy * oy - poles[:, 2:3] ** 2)
    tp = torch.where(disc >= 0, (-b - disc.clamp_min(0).sqrt()) / (2 * a), math.inf)
    zp = o[2] + tp * d[:, 2]
    best = torch.minimum(best, torch.where((tp > 1e-6) & (zp >= 0) & (zp <= poles[:, 3:4]), tp, math.inf).amin(0))
    keep = (best <= reach) & (torch.rand(best.shape, generator=gen, device=dev) >= 0.1)
    best = best + 0.02 * torch.randn(best.shape, generator=gen, device=dev, dtype=f64)
    world = o + best[keep, None] * d[keep]
    return ((world - t) @ R).float().contiguous()


def _thin(xyz, n, gen):
    """At most n points, in scan order (n = 0: all)."""
    if n == 0 or n >= xyz.shape[0]:
        return xyz
    pick = torch.randperm(xyz.shape[0], generator=gen, device=xyz.device)[:n].sort().values
    return xyz[pick].contiguous()


def _offset(rng, max_t, max_yaw):
    r, a = max_t * math.sqrt(rng.uniform()), rng.uniform(-math.pi, math.pi)
    return np.array([r * math.cos(a), r * math.sin(a), rng.uniform(-0.1, 0.1), math.radians(rng.uniform(-1, 1)),
                     math.radians(rng.uniform(-1, 1)), math.radians(rng.uniform(-max_yaw, max_yaw))])


def _pair(c, rng, gen):
    scene = _scene(rng)
    T = _offset(rng, c["half_xy"], c["half_yaw"])
    A = _thin(_scan(scene, np.zeros(6), c["beams"], c["az_deg"], gen), c["points"], gen)
    B = _thin(_scan(scene, T, c["beams"], c["az_deg"], gen), c["points"], gen)
    return A, B, T


# ---------------------------------------------------------------------------------------
# grids and poses
# ---------------------------------------------------------------------------------------
def _desc(c):
    res = c["res_mm"] / 1000.0
    return dict(origin=(-c["x"] * res / 2, -c["y"] * res / 2, Z_LOW), res_m=res, dims=(c["x"], c["y"], c["z"]),
                feature=c["feature"], count_levels=7, var_levels=8 if c["feature"] == JOINT else 15)


def _counts(c):
    return [int(m) for m in c["counts"].split("x")]


def _half(c):
    return np.array([c["half_xy"], c["half_xy"], 0.25, math.radians(1.0), math.radians(1.0),
                     math.radians(c["half_yaw"])])


def _lattice(centre, half, counts, order):
    """Candidate poses on a lattice around `centre`, the axes (0-2 t, 3-5 r) from slowest to fastest
    as `order` lists them."""
    axes = [np.array([x]) if m < 2 else x + np.linspace(-h, h, m) for x, h, m in zip(centre, half, counts)]
    order = [int(a) for a in order]
    g = np.meshgrid(*(axes[a] for a in order), indexing="ij")
    etas = np.empty((g[0].size, 6))
    for a, values in zip(order, g):
        etas[:, a] = values.reshape(-1)
    return etas


def _scatter(rng, n, centre, half):
    return centre + rng.uniform(-1.0, 1.0, (n, 6)) * half


def _near(rng, T, half):
    """An initial guess: the truth, off by up to half of each range."""
    return T + rng.uniform(-0.5, 0.5, 6) * half


def _round_poses(origin, etas):
    """Rows of 12 float32: R = Rz Ry Rx (FP64, rounded once) and t - origin."""
    cx, cy, cz = np.cos(etas[:, 3:6]).T
    sx, sy, sz = np.sin(etas[:, 3:6]).T
    R = [cz * cy, (cz * sy) * sx - sz * cx, (cz * sy) * cx + sz * sx,
         sz * cy, (sz * sy) * sx + cz * cx, (sz * sy) * cx - cz * sx, -sy, cy * sx, cy * cx]
    t = etas[:, :3] - np.asarray(origin, np.float32).astype(np.float64)
    return np.concatenate([np.stack(R, 1), t], 1).astype(np.float32)


def _inputs(c, seed):
    """What `prepare` and `exact` start from."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    kind = c["kind"]
    if kind == "batch":
        out = []
        base = [_pair(dict(c, points=0), rng, gen) for _ in range(2)]
        for i in range(c["n"]):
            A, B, T = base[i % 2]
            n = int(round(math.exp(rng.uniform(math.log(20000), math.log(110000)))))
            res = (250, 500, 1000)[i % 3]
            ci = dict(c, res_mm=res, x=80000 // res, y=80000 // res, z=8000 // res, feature=ZVAR)
            out.append((_desc(ci), _thin(A, n, gen), _thin(B, n, gen), _lattice(_near(rng, T, _half(c)), _half(c),
                                                                              _counts(c), c["order"])))
        return out
    if kind == "serve":
        refs, requests = [], []
        for k in range(4):
            A, B, T = _pair(dict(c, points=0), rng, gen)
            res = (250, 500, 750, 1000)[k]
            ci = dict(c, res_mm=res, x=80000 // res, y=80000 // res, z=8000 // res, feature=ZVAR)
            refs.append((_desc(ci), A))
            requests.append((B, T))
        todo = []
        for i in range(c["n"]):
            k = int(rng.integers(4))
            B, T = requests[k]
            n = int(round(math.exp(rng.uniform(math.log(10000), math.log(110000)))))
            todo.append((k, _thin(B, n, gen), _near(rng, T, _half(c))))
        return refs, todo
    A, B, T = _pair(c, rng, gen)
    etas = None
    if kind in ("lattice", "lattice_host"):
        etas = _lattice(_near(rng, T, _half(c)), _half(c), _counts(c), c["order"])
    elif kind in ("poses", "poses_device"):
        etas = _scatter(rng, c["poses"], T, _half(c))
    elif kind == "refine":
        etas = _scatter(rng, c["n"], T, _half(c))
    elif kind == "search":
        etas = _near(rng, T, _half(c))
    return A, B, etas


# ---------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------
def _grid(desc, A):
    L = align.align_create_grid(**desc)
    align.align_set_reference(L, A)
    return L


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": case}
    if kind == "batch":
        s["batch"] = align.align_batch_create()
        s["pairs"] = [(_grid(desc, A), B, etas) for desc, A, B, etas in _inputs(c, seed)]
        return s
    if kind == "serve":
        refs, todo = _inputs(c, seed)
        s["server"] = align.align_server_create(32 << 30, 3)
        ids = [align.align_server_add_reference(s["server"], A.cpu().numpy(), **desc) for desc, A in refs]
        s["todo"] = [(ids[k], B.cpu().numpy(), init) for k, B, init in todo]  # requests arrive in host memory
        return s
    A, B, etas = _inputs(c, seed)
    s.update(A=A, B=B, etas=etas, grid=_grid(_desc(c), A))
    if kind == "lattice_host":
        s["B"] = B.cpu().numpy()
    elif kind == "poses_device":
        s["poses"] = torch.from_numpy(_round_poses(_desc(c)["origin"], etas)).cuda()
        P, K = etas.shape[0], s["grid"].K
        s["out"] = (torch.empty(P, dtype=torch.float32, device="cuda"), torch.empty(1, dtype=torch.int64, device="cuda"),
                    torch.empty((P, K, K), dtype=torch.int32, device="cuda"))
    return s


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind in ("lattice", "lattice_host"):
        mi, best, _ = align.align_eval_mi(s["grid"], s["B"], eta6=s["etas"])
        return {"mi": mi, "best": best}
    if kind == "poses":
        mi, best, hist = align.align_eval_mi(s["grid"], s["B"], eta6=s["etas"], with_hist=True)
        return {"mi": mi, "best": best, "hist": hist.view(np.int32)}
    if kind == "poses_device":
        mi, best, hist = align.align_eval_mi(s["grid"], s["B"], poses12=s["poses"], out=s["out"])
        return {"mi": mi, "best": best, "hist": hist}
    if kind == "search":
        align.align_set_reference(s["grid"], s["A"])
        T, mi, level_best = align.align_search(s["grid"], s["B"], s["etas"], _half(c), levels=c["levels"],
                                               counts=_counts(c))
        return {"T": T, "mi": np.float32(mi), "level_best": level_best}
    if kind == "reference":
        align.align_set_reference(s["grid"], s["A"])
        symbols, box = align.align_get_reference(s["grid"])
        return {"symbols": symbols, "box": box}
    if kind == "batch":
        got = align.align_eval_batch(s["batch"], s["pairs"], graph=True)
        return {"mi": [mi for mi, _ in got], "best": [best for _, best in got]}
    if kind == "refine":
        T, mi, it = align.align_refine_nm(s["grid"], s["B"], s["etas"], step=0.25 * _half(c), max_iter=c["iters"])
        return {"T": T, "mi": mi, "iterations": it}
    tickets = [align.align_submit(s["server"], k, B, init, _half(c), levels=c["levels"], counts=_counts(c))
               for k, B, init in s["todo"]]
    got = [align.align_wait(s["server"], t) for t in tickets]
    return {"T": np.stack([r["T"] for r in got]), "mi": np.array([r["mi"] for r in got], np.float32),
            "status": np.array([r["status"] for r in got], np.int32)}


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------
def _symbols(feature):
    return 1 + (7 if feature == COUNT else 15 if feature == ZVAR else 56)


def work(case):
    """Bytes: scans, poses and A's symbols read once, results written once.  Operations: a
    rotation (15) per point and distinct rotation; the axis map (add, scale, floor) per point,
    rotation and axis sample on a lattice, or per point and pose (9) without one; the MI sums
    (4 K^2) per pose."""
    c, kind = case, case["kind"]
    rays = c["beams"] * int(round(360.0 / c["az_deg"]))
    N = c["points"] or int(rays * 0.87)
    V, K = c["x"] * c["y"] * c["z"], _symbols(c["feature"])
    m = _counts(c)
    P, n_rot, axes = _product(m), m[3] * m[4] * m[5], m[0] + m[1] + m[2]

    def lattice(N, V, K):
        return 12 * N + 48 * P + 4 * P + V, N * n_rot * (15 + 3 * axes) + P * 4 * K * K

    if kind in ("lattice", "lattice_host"):
        b, f = lattice(N, V, K)
    elif kind in ("poses", "poses_device", "refine"):
        n = c["poses"] if kind != "refine" else c["n"] * (7 + c["iters"])  # at least a reflection per iteration
        b = 12 * N + 52 * n + V + (4 * n * K * K if kind != "refine" else 0)
        f = n * (24 * N + 4 * K * K)
    elif kind == "search":
        b, f = 24 * N + V, c["levels"] * lattice(N, V, K)[1]
    elif kind == "reference":
        b, f = 12 * N + V, 24 * N
    else:  # batch, serve: 80 x 80 x 8 m grids, points log-uniform (means of 54k and 41k)
        res = (250, 500, 1000) if kind == "batch" else (250, 500, 750, 1000)
        Vm = sum((80000 // r) ** 2 * (8000 // r) for r in res) / len(res)
        n1, f1 = lattice(52800 if kind == "batch" else 41700, Vm, 16)
        b, f = c["n"] * n1, c["n"] * f1 * (1 if kind == "batch" else c["levels"])
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------------------
# the same in plain torch, sums in whole numbers and entropies in 64 bits
# ---------------------------------------------------------------------------------------
EXACT_MAX = 1.2e9  # points x poses


def _fma(a, b, c):
    return (a.double() * b.double() + c.double()).float()  # the product is exact in 64 bits


def _voxels(desc, R, t, xyz):
    """Voxel key (-1 outside) and z offset in mm of every point under translations t (P x 3) after
    rotation R: the method's FP32 map, operation by operation."""
    X, Y, Z = desc["dims"]
    inv = torch.tensor(np.float32(1.0 / float(np.float32(desc["res_m"]))), device="cuda")
    x, y, z = xyz.unbind(1)
    u = [_fma(R[3 * i], x, _fma(R[3 * i + 1], y, R[3 * i + 2] * z)) for i in range(3)]
    g = [u[i][None, :] + t[:, i:i + 1] for i in range(3)]
    k = [(gi * inv).floor() for gi in g]
    ok = (k[0] >= 0) & (k[0] < X) & (k[1] >= 0) & (k[1] < Y) & (k[2] >= 0) & (k[2] < Z)
    k = [torch.where(ok, ki, torch.zeros_like(ki)).long() for ki in k]
    dz = torch.where(ok, (g[2] * 1000.0).round(), torch.zeros_like(g[2])).long() - k[2] * int(round(desc["res_m"] * 1000))
    return torch.where(ok, (k[2] * Y + k[1]) * X + k[0], torch.full_like(k[0], -1)), dz


def _features(desc, key, dz):
    """(pose, voxel, symbol) of every occupied voxel."""
    V = desc["dims"][0] * desc["dims"][1] * desc["dims"][2]
    P = key.shape[0]
    ok = key >= 0
    at = (key + torch.arange(P, device="cuda")[:, None] * V)[ok]
    n = torch.zeros(P * V, dtype=torch.int32, device="cuda").index_add_(0, at, torch.ones_like(at, dtype=torch.int32))
    where = n.nonzero().squeeze(1)
    slot = n  # reuse: voxel -> its place in `where`
    n = n[where].long()
    slot[where] = torch.arange(where.numel(), dtype=torch.int32, device="cuda")
    at, d = slot[at].long(), dz[ok]
    s1, s2 = torch.zeros_like(n).index_add_(0, at, d), torch.zeros_like(n).index_add_(0, at, d * d)
    Lc, Lv = desc["count_levels"], desc["var_levels"]
    lc = sum((n >= (1 << (j + 1))).long() for j in range(Lc - 1))
    r2 = int(round(desc["res_m"] * 1000)) ** 2
    spread = n * s2 - s1 * s1
    lv = sum((spread >= (r2 >> (2 + Lv - 1 - j)) * n * n).long() for j in range(Lv - 1))
    sym = 1 + (lc if desc["feature"] == COUNT else lv if desc["feature"] == ZVAR else lc * Lv + lv)
    return where // V, where % V, sym


def _box(desc, pose, voxel, P):
    """Occupied box (lowest and highest voxel per axis) of every pose."""
    X, Y, _ = desc["dims"]
    lo = torch.full((P, 3), 1 << 30, dtype=torch.int64, device="cuda")
    hi = torch.full((P, 3), -1, dtype=torch.int64, device="cuda")
    k = torch.stack([voxel % X, (voxel // X) % Y, voxel // (X * Y)], 1)
    for a in range(3):
        lo[:, a].scatter_reduce_(0, pose, k[:, a], "amin")
        hi[:, a].scatter_reduce_(0, pose, k[:, a], "amax")
    return lo, hi


def _exact_mi(desc, A, B, poses):
    """(MI in 64 bits, joint histograms) of scan B under every row of `poses` (12 float32)."""
    X, Y, Z = desc["dims"]
    K = {COUNT: 1 + desc["count_levels"], ZVAR: 1 + desc["var_levels"],
         JOINT: 1 + desc["count_levels"] * desc["var_levels"]}[desc["feature"]]
    A, symA, boxA = _exact_reference(desc, A)
    sums = torch.zeros((K, Z + 1, Y + 1, X + 1), dtype=torch.int32, device="cuda")
    for q in range(K):
        one = (symA.reshape(Z, Y, X) == q).to(torch.int32)
        sums[q, 1:, 1:, 1:] = one.cumsum(0, dtype=torch.int32).cumsum(1, dtype=torch.int32).cumsum(2, dtype=torch.int32)
    P = poses.shape[0]
    mi, hist = torch.zeros(P, dtype=torch.float64), torch.zeros((P, K, K), dtype=torch.int64)
    step = max(1, min(int(6e7 // (X * Y * Z)), int(3e7 // max(1, B.shape[0])), 256))
    turn = np.lexsort(poses[:, :9].T)  # poses of one rotation together
    p12 = torch.from_numpy(poses[turn]).cuda()
    same = (p12[1:, :9] == p12[:-1, :9]).all(1).cpu().numpy()
    a = 0
    while a < P:
        b = a + 1
        while b < P and b - a < step and same[b - 1]:
            b += 1
        key, dz = _voxels(desc, p12[a, :9], p12[a:b, 9:], B)
        pose, voxel, symB = _features(desc, key, dz)
        lo, hi = _box(desc, pose, voxel, b - a)
        lo, hi = torch.maximum(lo, boxA[:3]), torch.minimum(hi, boxA[3:])
        k = torch.stack([voxel % X, (voxel // X) % Y, voxel // (X * Y)], 1)
        inside = ((k >= lo[pose]) & (k <= hi[pose])).all(1)
        h = torch.bincount((pose * K * K + symA[voxel] * K + symB)[inside], minlength=(b - a) * K * K)
        h = h.reshape(b - a, K, K)
        empty = (lo > hi).any(1)
        (x0, y0, z0), (x1, y1, z1) = (torch.where(empty[:, None], torch.zeros_like(e), e).unbind(1) for e in (lo, hi + 1))
        # A's voxels of every symbol in the box, from its summed volumes
        nA = (sums[:, z1, y1, x1] - sums[:, z0, y1, x1] - sums[:, z1, y0, x1] - sums[:, z1, y1, x0] +
              sums[:, z0, y0, x1] + sums[:, z0, y1, x0] + sums[:, z1, y0, x0] - sums[:, z0, y0, x0]).T.long()
        h[:, :, 0] = nA - h.sum(2)  # where B has no voxel
        h[empty] = 0
        N = h.sum((1, 2)).clamp_min(1).double()

        def entropy(c):
            q = c.double() / N.reshape(-1, *([1] * (c.dim() - 1)))
            return -torch.where(q > 0, q * q.clamp_min(1e-300).log(), torch.zeros_like(q)).flatten(1).sum(1)

        mi[turn[a:b]] = (entropy(h.sum(2)) + entropy(h.sum(1)) - entropy(h)).cpu()
        hist[turn[a:b]] = h.cpu()
        a = b
    return mi, hist


def _exact_reference(desc, A):
    V = desc["dims"][0] * desc["dims"][1] * desc["dims"][2]
    p = torch.from_numpy(_round_poses(desc["origin"], np.zeros((1, 6)))).cuda()
    pose, voxel, sym = _features(desc, *_voxels(desc, p[0, :9], p[:, 9:], A))
    symA = torch.zeros(V, dtype=torch.int64, device="cuda")
    symA[voxel] = sym
    lo, hi = _box(desc, pose, voxel, 1)
    return A, symA, torch.cat([lo[0], hi[0]])


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind not in ("lattice", "lattice_host", "poses", "poses_device", "reference", "batch"):
        return None  # a search's or an optimiser's path hangs on every choice before it
    got = _inputs(c, seed)
    if kind == "batch":
        if sum(B.shape[0] * etas.shape[0] for _, _, B, etas in got) > 3 * EXACT_MAX:
            return None
        mi = [_exact_mi(desc, A, B, _round_poses(desc["origin"], etas))[0] for desc, A, B, etas in got]
        return {"mi": mi, "best": [None] * len(mi)}
    A, B, etas = got
    desc = _desc(c)
    if kind == "reference":
        _, symA, box = _exact_reference(desc, A)
        return {"symbols": symA.to(torch.uint8), "box": box.to(torch.int32)}
    if B.shape[0] * float(etas.shape[0]) > EXACT_MAX:
        return None
    mi, hist = _exact_mi(desc, A, B, _round_poses(desc["origin"], etas))
    out = {"mi": mi, "best": None}
    if kind in ("poses", "poses_device"):
        out["hist"] = hist.to(torch.int32)
    return out
