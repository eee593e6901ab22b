"""The work that programs have this library do, as cases to be timed.

A case names a use of the library (`kind`), a scene and its sizes. Scans come
from the package's own generators: the single-frame scene (sphere, wall,
slotted plate), the pine seen from an orbiting rosette sensor, three pines,
and the pine at the large map's resolution (1 cm, 512 directions). Maps are
warm, as a stream's are: all scans but the first are integrated beforehand, so
a first pass also meets bricks that the map has not seen.

`exact` restates the integration and the soft clearance in 64 bits with plain
torch for the cases whose results are computed numbers; labels, directions and
voxel words are whole numbers and have none.
"""
import functools
import math

import numpy as np
import torch

from paper_2608_06412_gb300 import af, synth, workload

HEMISPHERE = 64       # orientations per point of the soft field
REFINE_STEPS = 20
#: Voxels of a scene that a sensor sees, about: n returns hit
#: SEEN (1 - exp(-n / SEEN)) of them.
SEEN = {"plate": 4500, "pine": 21000, "forest": 80000, "pine_1cm": 180000}


def listed():
    return [
        # a short-range sensor's packet of a few hundred returns, handled as it
        # comes: latency and launches are all there is
        dict(name="frame_packet", kind="frame", scene="plate", n=503, scans=3, K=32, table="sphere", signed=False),
        # the single-frame scene from pinned host buffers, copies included: the
        # call a sensor driver makes when it needs the labels now
        dict(name="frame_host", kind="host", scene="plate", n=20000, scans=3, K=32, table="sphere", signed=False),
        # one 10 Hz frame of the pine stream: integrate, score its points
        dict(name="frame_pine", kind="frame", scene="pine", n=20000, scans=3, K=64, table="sphere", signed=False),
        # a dense sensor in a small forest, the largest tool, 256 directions
        dict(name="frame_forest", kind="frame", scene="forest", n=59999, scans=2, K=128, table="sphere", signed=False),
        # a change of tool: every surface point of a 1 cm map is scored again
        dict(name="score_map_1cm", kind="score", scene="pine_1cm", n=40001, scans=3, K=256, table="sphere", signed=False),
        # several robots ticked together, uneven scenes
        dict(name="batch_tick", kind="batch", scenes=10, n_lo=2000, n_hi=16000),
        # the stateful layer: six frames of the stream, then the points read out
        dict(name="layer_frames", kind="layer", scene="pine", n=20000, scans=6, K=64, table="sphere", signed=False,
             budget=16384, sample=256, exact_trigger=True, c2f=False),
        # refinement in the loop: a scan arrives, its points are scored and the
        # accessible ones refined on the map as it is now
        dict(name="refine_online", kind="online", scene="pine", n=20000, scans=3, K=64, table="sphere", signed=False),
        # refinement of every accessible point of a finished map, from its best
        # direction
        dict(name="refine_map", kind="refine", scene="pine", n=20000, scans=6, K=64, table="sphere", signed=False),
        # the soft field over all orientations of every point: planning over a
        # finished map
        dict(name="soft_field", kind="field", scene="pine", n=20000, scans=6, K=64, table="sphere", signed=False),
        # a caller's own optimiser: forward and backward through autograd
        dict(name="soft_gradient", kind="grad", scene="pine", n=20000, scans=3, K=64, table="sphere", signed=False,
             per_point=4),
        # the call for programs that may not allocate: a scan into their box
        dict(name="box_scan", kind="box", scene="pine", n=20000, scans=3, K=64, table="sphere", signed=False),
    ]


#: What the stateful layer exports per point.
LAYER_FIELDS = [("ijk", (3,), np.int32), ("normal", (3,), np.float32), ("label", (), np.uint8),
                ("score", (), np.int16), ("best", (), np.int16), ("a", (), np.float32),
                ("queued", (), np.uint8), ("nviews", (), np.int32)]


#: The dense voxel box that a program without an allocator keeps for a scene,
#: from the low corner of the scene's map box.
BOX = {"plate": (224, 128, 176), "pine": (400, 400, 680), "forest": (640, 640, 680)}


def _point_count(case):
    """Surface points of a call: those of one scan, or of a finished map."""
    n, N = case["n"], SEEN[case["scene"]]
    if case["kind"] in ("score", "refine", "field", "grad"):
        n, N = n * case["scans"], 1.5 * N   # the sensor moved between the scans
    return max(1, int(0.95 * N * (1 - math.exp(-n / N))))


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "host", "score", "batch", "layer", "online",
                       "refine", "field", "grad", "box"])
    if kind == "batch":
        lo = rng.randint(300, 4000)
        return dict(kind=kind, scenes=rng.randint(2, 10), n_lo=lo, n_hi=rng.randint(lo + 1, 16000))
    # the online step writes a view of the whole map box, the forest's the largest
    scene = rng.choice(["plate", "pine", "pine", "pine" if kind == "online" else "forest"])
    if kind == "score" and rng.random() < 0.5:
        scene = "pine_1cm"
    top = {"frame": 59999, "box": 40000, "online": 20000}.get(kind, 20000)
    ring = rng.random() < 0.25      # the paper's yaw ring and 70 degree cone
    c = dict(kind=kind, scene=scene, n=_log_int(rng, 300, top), scans=rng.randint(2, 4),
             K=90 if ring else rng.choice([16, 32, 64, 128]),
             table="ring" if ring else "sphere", signed=rng.random() < 0.2)
    if kind == "grad":
        c["per_point"] = rng.randint(1, 6)
    if kind == "layer":
        c.update(budget=_log_int(rng, 200, 131072), sample=rng.choice([256, 256, 64, 0]),
                 exact_trigger=rng.random() < 0.7, c2f=ring)
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _workload(scene, seed):
    """Scene, map box and parameters of one of the scenes, tool included."""
    if scene == "plate":
        return workload.single_frame(seed)
    if scene == "pine":
        return workload.pine_stream(seed)
    p = dict(synth.LARGE_MAP if scene == "pine_1cm" else synth.PINE_STREAM)
    p["seed"] = seed
    if scene == "forest":
        p["tool"] = dict(workload.BATCH_TOOLS[2])
        p["orbit_radius"] = 5.5
        sc = workload.forest_scene(seed, 3)
    else:
        sc = synth.pine_scene(seed)
    r = p["orbit_radius"] + 0.5
    lo = np.minimum(sc.lo, [-r, -r, 0.0])
    hi = np.maximum(sc.hi, [r, r, p["orbit_height"]])
    dmin, db = synth.domain_bricks(lo, hi, p["v"], margin=0.5)
    return workload.Workload(scene, p, sc, dmin, db, synth.fibonacci_dirs(2 * p["K"]))


@functools.lru_cache(maxsize=96)
def _scans(scene, seed, n, scans):
    """The workload and `scans` scans of n returns from a moving sensor: (returns
    in the sensor frame, pose, surface points, normals), numpy arrays."""
    W = _workload(scene, seed)
    p, out = W.params, []
    for k in range(scans):
        if scene == "plate":
            f = synth.cone_frame(W.scene, n, p["sigma"], seed + 7919 * k,
                                 origin=(0.0, 0.06 * k, 0.03 * k))
        else:   # a twelfth of an orbit between scans: some bricks new, most seen
            f = synth.rosette_frame(W.scene, 25 * k, seed, n_hits=n, sigma=p["sigma"],
                                    orbit_radius=p["orbit_radius"],
                                    orbit_height=p["orbit_height"], frames_per_orbit=300)
        out.append((f.pts, f.pose, *synth.surface_points(f.world, f.normal, p["v"])))
    return W, out


def _table(case, W):
    """The tool and the direction table: the Fibonacci sphere, or the paper's yaw
    ring with its 70 degree cone."""
    tool = W.af_tool()
    if case["table"] == "ring":
        tool.cos_theta_max = synth.COS_70
        return tool, synth.yaw_ring(180)
    return tool, synth.fibonacci_dirs(2 * case["K"])


def _caps(case):
    big = case["scene"] == "pine_1cm" or case["scene"] == "forest"
    return dict(hash_capacity=1 << (19 if big else 18), pool_blocks=1 << (18 if big else 17),
                max_returns=1 << 16, max_points=1 << 16, clamp_signed=int(case["signed"]))


def _cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _map_points(case, scans, v):
    """Points and normals of a finished map: one per voxel over all scans, first
    occurrence, as many as the case scores."""
    pts = np.concatenate([s[2] for s in scans])
    nrm = np.concatenate([s[3] for s in scans])
    ijk = np.floor(pts.astype(np.float64) / np.float64(np.float32(v))).astype(np.int64)
    _, first = np.unique(ijk, axis=0, return_index=True)
    first = np.sort(first)
    return _take((pts[first], nrm[first]), _point_count(case))


def _parameters(n, seed):
    """Tangent offsets and standoffs of n pairs in mid-optimisation, and the
    weights of the caller's loss."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    par = [torch.randn(n, generator=g, device="cuda") * 0.05 for _ in range(2)]
    par.append(torch.rand(n, generator=g, device="cuda") * 0.03)
    return par, torch.rand(n, generator=g, device="cuda")


def _take(points, count):
    """`count` of the points and normals, evenly spaced in their order."""
    at = np.arange(count) * len(points[0]) // count
    return tuple(np.ascontiguousarray(a[at]) for a in points)


def _prepare_batch(case, seed):
    maps, items = [], []
    S = workload.batch_scenes(case["scenes"], seed % 100000, case["n_lo"], case["n_hi"])
    for i, W in enumerate(S):
        p = W.params
        n = case["n_lo"] + (case["n_hi"] - case["n_lo"]) * i // (len(S) - 1)
        f = synth.rosette_frame(W.scene, 0, p["seed"], n_hits=n, sigma=p["sigma"],
                                orbit_radius=p["orbit_radius"], orbit_height=p["orbit_height"],
                                frames_per_orbit=300)
        m = af.Map(W.af_config(hash_capacity=1 << 17, pool_blocks=1 << 16, max_returns=1 << 16,
                               max_points=1 << 16))
        m.set_tool(W.af_tool(), W.dirs)
        # two scans of a standing sensor: the even and the odd returns
        pair = []
        for k in range(2):
            pts, nrm = _take(synth.surface_points(f.world[k::2], f.normal[k::2], p["v"]), n * 2 // 5)
            pair.append((_cuda(f.pts[k::2]), f.pose, _cuda(pts), _cuda(nrm)))
        m.integrate_scan(pair[1][0], pair[1][1])
        maps.append(m)
        items.append(pair)
    ticks = []
    for k in range(2):
        m = sum(len(it[k][2]) for it in items)
        label = torch.zeros(m, dtype=torch.uint8, device="cuda")
        best = torch.zeros(m, dtype=torch.int16, device="cuda")
        tick, label_at = [], 0
        for it in items:
            x, pose, pts, nrm = it[k]
            end = label_at + len(pts)
            tick.append((x, pose, pts, nrm, label[label_at:end], best[label_at:end]))
            label_at = end
        ticks.append((tick, label, best))
    return dict(case=case, batch=af.Batch(maps), ticks=ticks, k=0)


def prepare(case, seed):
    if case["kind"] == "batch":
        return _prepare_batch(case, seed)
    kind = case["kind"]
    W, scans = _scans(case["scene"], seed, case["n"], case["scans"])
    p = W.params
    s = dict(case=case, k=0, v=p["v"])
    cfg = W.af_config(**_caps(case))
    scans = [(x, pose, *_take(points, _point_count(case))) for x, pose, *points in scans]
    s["scans"] = [(_cuda(x), pose, _cuda(pts), _cuda(nrm)) for x, pose, pts, nrm in scans]
    if kind == "box":   # cleared once, as its owner does
        s["cfg"] = cfg
        s["box_min"] = np.array(W.dom_min) * 8
        s["box_dim"] = np.array(BOX[case["scene"]])
        count = int(np.prod(s["box_dim"]))
        s["vox"] = torch.zeros(count, dtype=torch.int64, device="cuda")
        s["flags"] = torch.zeros(count, dtype=torch.uint8, device="cuda")
        for x, pose, _, _ in s["scans"][1:]:
            af.integrate_scan_noalloc(cfg, x, pose, s["box_min"], s["box_dim"], s["vox"], s["flags"])
        return s
    m = af.Map(cfg)
    tool, dirs = _table(case, W)
    m.set_tool(tool, dirs)
    s["map"] = m
    if kind == "layer":
        c2f = dict(c2f_stride=10, c2f_half=12, c2f_radius=0.3) if case["c2f"] else {}
        m.points_enable(af.PointsConfig(trig_tsdf=2 * p["v"], capacity=1 << 20, budget=case["budget"],
                                        trig_sample=case["sample"],
                                        trig_exact=int(case["exact_trigger"]), **c2f))
        # the reader's own arrays, room for a point per return
        s["field"] = {k: np.zeros((case["n"] * case["scans"], *t), d) for k, t, d in LAYER_FIELDS}
        return s
    finished = kind in ("score", "refine", "field", "grad")
    # a finished map has seen each scan three times; a stream's all but the next
    for x, pose, _, _ in (s["scans"] * 3 if finished else s["scans"][1:]):
        m.integrate_scan(x, pose)
    if finished:
        pts, nrm = _map_points(case, _scans(case["scene"], seed, case["n"], case["scans"])[1], p["v"])
        s["pts"], s["nrm"] = _cuda(pts), _cuda(nrm)
    if kind == "host":
        pin = lambda a: torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()  # noqa: E731
        s["host"] = [(pin(x), pose, pin(pts), pin(nrm)) for x, pose, pts, nrm in scans]
        s["label"] = pin(np.zeros(_point_count(case), np.uint8))
        s["best"] = pin(np.zeros(_point_count(case), np.int16))
    if kind == "refine":
        s["u0"] = m.soft_start(*m.score(s["pts"], s["nrm"]))
    if kind == "field":
        s["table"] = synth.fibonacci_hemisphere(HEMISPHERE, tool.cos_theta_max)
        n = len(s["pts"]) * HEMISPHERE
        s["u0"] = torch.empty((n, 3), device="cuda")
        s["zero"] = torch.zeros(n, device="cuda")
    if kind == "grad":
        s["u0"] = m.soft_seed(s["nrm"], synth.fibonacci_hemisphere(case["per_point"], 0.3))
        par, s["weight"] = _parameters(len(s["u0"]), seed)
        s["par"] = [t.requires_grad_() for t in par]
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(s):
    kind = s["case"]["kind"]
    k = s["k"]
    if kind == "batch":
        s["k"] = (k + 1) % len(s["ticks"])
        tick, label, best = s["ticks"][k]
        s["batch"].tick(tick)
        return label, best
    s["k"] = (k + 1) % len(s["scans"])
    x, pose, pts, nrm = s["scans"][k]
    if kind == "box":
        af.integrate_scan_noalloc(s["cfg"], x, pose, s["box_min"], s["box_dim"], s["vox"], s["flags"])
        return s["vox"], s["flags"]
    m = s["map"]
    if kind == "frame":
        m.integrate_scan(x, pose)
        return m.score(pts, nrm)
    if kind == "host":
        x, pose, pts, nrm = s["host"][k]
        m.frame_host(x, pose, pts, nrm, s["label"], s["best"])
        return s["label"], s["best"]
    if kind == "score":
        return m.score(s["pts"], s["nrm"])
    if kind == "layer":
        for x, pose, _, _ in s["scans"]:
            m.points_frame(x, pose)
        for name, a in m.points_export().items():
            s["field"][name][:len(a)] = a
        return s["field"]
    if kind == "online":
        m.integrate_scan(x, pose)
        label, best = m.score(pts, nrm)
        u0 = m.soft_start(label, best)
        a, b, h = (torch.zeros(len(pts), device="cuda") for _ in range(3))
        c, cmin = m.soft_refine(pts, u0, a, b, h, 1, steps=REFINE_STEPS)
        return label, best, a, b, h, c, cmin
    if kind == "refine":
        a, b, h = (torch.zeros(len(s["pts"]), device="cuda") for _ in range(3))
        c, cmin = m.soft_refine(s["pts"], s["u0"], a, b, h, 1, steps=REFINE_STEPS)
        return a, b, h, c, cmin
    if kind == "field":
        m.soft_seed(s["nrm"], s["table"], out=s["u0"])
        c = m.soft_clearance_raw(s["pts"], s["u0"], s["zero"], s["zero"], s["zero"], HEMISPHERE)
        return (c, *m.soft_best(c, HEMISPHERE, u0=s["u0"]))
    c = m.soft_clearance(s["pts"], s["u0"], *s["par"], s["case"]["per_point"])
    return (c.detach(), *torch.autograd.grad(c, s["par"], s["weight"]))


def work(case):
    """Bytes: each return, point, normal and result once, each touched voxel word
    read and written once. Operations: 41 per (return, cube voxel) pair as the
    method states them, 6 per direction's normal test, 40 per axis sample of a
    soft clearance (90 with its gradient)."""
    kind = case["kind"]
    if kind == "batch":
        n = case["scenes"] * (case["n_lo"] + case["n_hi"]) // 4
        m, cube, K, samples, touched = 0.8 * n, 343, 70, 62, 30 * n
    else:
        fine = case["scene"] == "pine_1cm"
        n, m = case["n"], _point_count(case)
        cube, K, samples = (729 if fine else 343), case["K"], (175 if fine else 62)
        touched = 30 * n
    scan = dict(bytes=12 * n + 16 * touched, flops=41 * n * cube)
    score = dict(bytes=27 * m, flops=6 * m * 2 * K)
    if kind == "box":
        return scan
    if kind in ("frame", "host", "batch"):
        return dict(bytes=scan["bytes"] + score["bytes"], flops=scan["flops"] + score["flops"])
    if kind == "score":
        return dict(bytes=27 * m, flops=6 * m * 2 * K)
    if kind == "layer":
        f = case["scans"]
        return dict(bytes=f * (scan["bytes"] + 64 * m), flops=f * (scan["flops"] + score["flops"]))
    if kind == "online":
        return dict(bytes=scan["bytes"] + score["bytes"] + 56 * m,
                    flops=scan["flops"] + score["flops"] + m * samples * (90 * REFINE_STEPS + 40))
    if kind == "refine":
        return dict(bytes=56 * m, flops=m * samples * (90 * REFINE_STEPS + 40))
    if kind == "field":
        return dict(bytes=24 * m + m * HEMISPHERE * 16 + 20 * m,
                    flops=m * HEMISPHERE * samples * 40)
    pairs = m * case["per_point"]
    return dict(bytes=24 * m + 44 * pairs, flops=pairs * samples * 130)


# ---------------------------------------------------------------------------
# 64-bit restatement
# ---------------------------------------------------------------------------

def _field64(W, scans, signed):
    """The TSDF of the map box after each of `scans` three times over (their mean
    is that of once): a dense (Z, Y, X) float64 tensor, tau where nothing was
    seen, one voxel of tau around the box."""
    p = W.params
    v, tau, m = float(np.float32(p["v"])), float(np.float32(p["tau"])), p["cube_radius"]
    lo = torch.tensor(W.dom_min, device="cuda") * 8
    dim = torch.tensor(W.dom_bricks, device="cuda") * 8
    X, Y, Z = (int(d) for d in dim)
    S = torch.zeros(X * Y * Z, dtype=torch.float64, device="cuda")
    w = torch.zeros_like(S)
    r = torch.arange(-m, m + 1, device="cuda")
    off = torch.stack(torch.meshgrid(r, r, r, indexing="ij"), -1).reshape(-1, 3)
    for xyz, pose, _, _ in scans:
        T = torch.from_numpy(pose).cuda().double()
        q = T[:3, 3]
        P = torch.from_numpy(xyz).cuda().double() @ T[:3, :3].T + q
        for c in P.split(4096):
            b = c - q
            rng = b.norm(dim=1)
            rel = torch.floor(c / v).long() - lo
            ok = (rng >= p["range_min"]) & (rng <= p["range_max"])
            ok &= ((rel >= m) & (rel + m < dim)).all(1)
            c, b, rng, rel = c[ok], b[ok], rng[ok], rel[ok]
            j = rel[:, None] + off
            x = ((j + lo).double() + 0.5) * v
            a = x - c[:, None]
            an = a.norm(dim=2)
            cos = (a * b[:, None]).sum(2) / (an * rng[:, None])
            keep = (an == 0) | (cos <= float(np.float32(p["cone_cos"])))
            d = (rng[:, None] - (x - q).norm(dim=2)).clamp(-tau if signed else 0.0, tau)
            at = ((j[..., 2] * Y + j[..., 1]) * X + j[..., 0])[keep]
            S.index_add_(0, at, d[keep])
            w.index_add_(0, at, torch.ones_like(d[keep]))
    D = torch.where(w > 0, S / w.clamp(min=1), torch.full_like(S, tau)).view(Z, Y, X)
    return torch.nn.functional.pad(D, (1, 1, 1, 1, 1, 1), value=tau), lo - 1, v, tau


def _basis64(n):
    s = torch.where(n[:, 2] >= 0, 1.0, -1.0).double()
    a = -1.0 / (s + n[:, 2])
    b = n[:, 0] * n[:, 1] * a
    t1 = torch.stack([1 + s * n[:, 0] ** 2 * a, s * b, -s * n[:, 0]], 1)
    return t1, torch.stack([b, s + n[:, 1] ** 2 * a, -n[:, 1]], 1)


def _clearance64(F, tool, pts, u0, a, b, h):
    """(C, hard clearance) of pairs, differentiable in a, b, h."""
    D, lo, v, tau = F
    f32 = np.float32
    J = int(math.floor(f32(f32(tool.length) + f32(tool.corr_length)) / f32(v)))
    js = [j for j in range(1, J + 1) if f32(j) * f32(v) > f32(tool.self_excl)]
    mar = torch.tensor([float(f32(tool.radius if f32(j) * f32(v) <= f32(tool.length) else tool.corr_radius))
                        for j in js], dtype=torch.float64, device="cuda")
    t1, t2 = _basis64(u0)
    q = u0 + a[:, None] * t1 + b[:, None] * t2
    u = q / q.norm(dim=1, keepdim=True)
    t = h[:, None] + torch.tensor(js, dtype=torch.float64, device="cuda") * v
    g = (pts[:, None] + t[..., None] * u[:, None]) / v - 0.5
    cell = torch.floor(g.detach())
    f = g - cell
    cell = cell.long() - lo
    Z, Y, X = D.shape
    hi = torch.tensor([X - 1, Y - 1, Z - 1], device="cuda")
    inside = ((cell >= 0) & (cell < hi)).all(-1)
    cell = torch.minimum(cell.clamp(min=0), hi - 1)
    flat = D.reshape(-1)
    at = (cell[..., 2] * Y + cell[..., 1]) * X + cell[..., 0]
    val = 0.0
    for k in range(8):
        wk = 1.0
        for i, bit in enumerate((k & 1, (k >> 1) & 1, k >> 2)):
            wk = wk * (f[..., i] if bit else 1 - f[..., i])
        val = val + wk * flat[at + (k & 1) + ((k >> 1) & 1) * X + (k >> 2) * X * Y]
    phi = torch.where(inside, val, torch.full_like(val, tau)) - mar
    ts = float(np.float32(af.TAU_S))
    return -ts * torch.logsumexp(-phi / ts, 1), phi.min(1).values


def _with_grad64(F, tool, pts, u0, a, b, h):
    with torch.enable_grad():
        par = [t.detach().requires_grad_() for t in (a, b, h)]
        c, cmin = _clearance64(F, tool, pts, u0, *par)
        return c.detach(), cmin.detach(), torch.autograd.grad(c.sum(), par)


@torch.no_grad()
def exact(case, seed):
    kind = case["kind"]
    if kind not in ("refine", "field", "grad"):
        return None
    W, scans = _scans(case["scene"], seed, case["n"], case["scans"])
    tool, _ = _table(case, W)
    F = _field64(W, scans, case["signed"])
    pts, nrm = (torch.from_numpy(t).cuda().double() for t in _map_points(case, scans, W.params["v"]))
    out = []
    if kind == "refine":
        u0 = prepare(case, seed)["u0"].double()   # NaN where there is no start
        for s, u in zip(pts.split(16384), u0.split(16384)):
            a, b, h = (torch.zeros(len(s), dtype=torch.float64, device="cuda") for _ in range(3))
            for _ in range(REFINE_STEPS):
                _, _, (ga, gb, gh) = _with_grad64(F, tool, s, u, a, b, h)
                a, b, h = a + 0.05 * ga, b + 0.05 * gb, (h + 0.005 * gh).clamp(0.0, 0.05)
            out.append((a, b, h, *_clearance64(F, tool, s, u, a, b, h)))
        # a trajectory parts from its neighbour at a kink of the field that rounding
        # puts it on either side of, so the offsets have no one value
        a, b, h, c, cmin = (torch.cat(t) for t in zip(*out))
        none = torch.isnan(a)
        return [None, None, h, c.masked_fill(none, math.nan), cmin.masked_fill(none, math.nan)]
    per = HEMISPHERE if kind == "field" else case["per_point"]
    e = torch.from_numpy(synth.fibonacci_hemisphere(
        per, tool.cos_theta_max if kind == "field" else 0.3)).cuda().double()
    if kind == "field":
        for s, u in zip(pts.split(512), nrm.split(512)):
            t1, t2 = _basis64(u)
            d = e[:, 0:1] * t1[:, None] + e[:, 1:2] * t2[:, None] + e[:, 2:3] * u[:, None]
            z = torch.zeros(len(s) * per, dtype=torch.float64, device="cuda")
            out.append(_clearance64(F, tool, s.repeat_interleave(per, 0), d.reshape(-1, 3), z, z, z)[0])
        c = torch.cat(out)
        return [c, None, c.view(-1, per).max(1).values, None]
    par, weight = _parameters(len(pts) * per, seed)
    a, b, h = (t.double() for t in par)
    t1, t2 = _basis64(nrm)
    d = (e[:, 0:1] * t1[:, None] + e[:, 1:2] * t2[:, None] + e[:, 2:3] * nrm[:, None]).reshape(-1, 3)
    pp = pts.repeat_interleave(per, 0)
    for i in range(0, len(d), 16384):
        j = slice(i, i + 16384)
        c, _, g = _with_grad64(F, tool, pp[j], d[j], a[j], b[j], h[j])
        out.append((c, *(x * weight[j].double() for x in g)))
    return [torch.cat(t) for t in zip(*out)]
