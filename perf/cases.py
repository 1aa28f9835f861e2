"""The work that users of the library have it do, as measurable cases.

Frames are synthetic, with the sizes and distributions of the workloads in
paper_2012_12618_gb300/synth.py (drawn here on the GPU, so that inputs are
made quickly): azimuth uniform in +-60 deg, |v| uniform in 0..40 m/s, a fixed
share of micro-Doppler outliers, Gaussian Doppler noise.  Every case goes
through the public binding of the C ABI, on one context and one stream, as a
program that estimates frame after frame does.

A case's cluster sizes follow from the case alone (so that outputs have one
shape); their order and every value follow from the seed.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2012_12618_gb300 import rvh

DEG = math.pi / 180.0
TAU = 0.1            # m/s, the inlier threshold of every workload
EPS, MIN_PTS = 1.0, 4  # DBSCAN radius (m) and core size of the scene workload
COUNTERS = ("inlier_count", "best_hypothesis", "status", "inlier_mask")


# ---- the cases ---------------------------------------------------------------------------

def estimate(name, clusters, law, lo, hi, dim, trials, outliers, sigma, band=0.0, memory="device", refine=0,
             confidence=0.0, line=False):
    return {"name": name, "entry": "estimate", "clusters": clusters, "law": law, "lo": lo, "hi": hi, "dim": dim,
            "trials": trials, "outliers": outliers, "sigma": sigma, "band": band, "memory": memory,
            "refine": refine, "confidence": confidence, "line": line}


def listed():
    return [
        # one frame of one radar with few objects: the smallest call, latency
        estimate("frame64", 64, "uniform", 16, 128, 2, 256, 0.20, 0.05),
        # one frame of a 2D radar of the serving load (50..2000 clusters), mean size
        estimate("radar2d", 1025, "loguniform", 8, 2048, 2, 256, 0.20, 0.05),
        # one frame of a 3D radar of the serving load: clusters beyond the shared-memory rows, two trial chunks
        estimate("radar3d", 1025, "loguniform", 8, 2048, 3, 2048, 0.25, 0.05),
        # the dense traffic frame, the headline workload
        estimate("dense2d", 4096, "loguniform", 8, 2048, 2, 1024, 0.20, 0.05),
        # many middling clusters with many outliers and points next to the threshold
        estimate("stress2d", 16384, "uniform", 32, 512, 2, 1024, 0.40, 0.08, band=0.05),
        # 3D velocities, the largest workload
        estimate("dense3d", 8192, "uniform", 24, 1024, 3, 2048, 0.25, 0.05),
        # the dense frame from page-locked host memory and back: a caller without device buffers
        estimate("dense2d_host", 4096, "loguniform", 8, 2048, 2, 1024, 0.20, 0.05, memory="pinned"),
        # the dense frame with the adaptive trial count
        estimate("dense2d_adaptive", 4096, "loguniform", 8, 2048, 2, 1024, 0.20, 0.05, confidence=0.99),
        # the dense frame with local-optimisation rounds after the refine
        estimate("dense2d_local_opt", 4096, "loguniform", 8, 2048, 2, 1024, 0.20, 0.05, refine=2),
        # Alg. 1 as printed: line fits with a MAD threshold
        estimate("dense2d_line", 4096, "loguniform", 8, 2048, 2, 1024, 0.20, 0.05, line=True),
        # a raw point cloud to velocities: DBSCAN, gather, estimate
        {"name": "scene", "entry": "scene", "objects": 512, "lo": 8, "hi": 1024, "range": 400.0, "trials": 1024},
        # eight radars' frames, 2D and 3D in turn, through the request queue
        {"name": "serving8", "entry": "serving", "frames": 8, "clusters": 1025, "lo": 8, "hi": 2048,
         "trials2d": 256, "trials3d": 2048},
    ]


def log_int(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    """One more case: any entry, sizes over the whole range, at most the largest listed case's cost."""
    kind = rng.choice(["estimate"] * 8 + ["scene", "scene", "serving"])
    if kind == "scene":
        # the field of view holds a little over one object per 10 m cell
        return {"entry": "scene", "objects": log_int(rng, 24, 512), "lo": 8, "hi": log_int(rng, 100, 1024),
                "range": 400.0, "trials": log_int(rng, 128, 1024)}
    if kind == "serving":
        return {"entry": "serving", "frames": rng.randint(2, 8), "clusters": log_int(rng, 50, 1025), "lo": 8,
                "hi": log_int(rng, 200, 2048), "trials2d": log_int(rng, 128, 1024),
                "trials3d": log_int(rng, 256, 2048)}
    flavour = rng.choice(["plain"] * 5 + ["adaptive", "local", "line", "host"])
    dim = 2 if flavour == "line" else rng.choice([2, 3])
    lo = log_int(rng, 8, 64)
    c = estimate("", log_int(rng, 24, 16384), rng.choice(["uniform", "loguniform"]), lo, log_int(rng, 2 * lo, 2048),
                 dim, log_int(rng, 128, 2048), rng.choice([0.1, 0.2, 0.25, 0.4]), rng.choice([0.03, 0.05, 0.08]),
                 memory=rng.choice(["pinned", "pageable"]) if flavour == "host" else "device",
                 refine=rng.randint(1, 4) if flavour == "local" else 0,
                 confidence=rng.choice([0.9, 0.99]) if flavour == "adaptive" else 0.0, line=flavour == "line")
    del c["name"]
    # line fits and rounds cost several times a plain trial, the listed ones included
    most = 1.2e9 if flavour in ("line", "local") else 4e9
    while pairs(c) * (c["dim"] - 1) > most and c["clusters"] > 24:
        c["clusters"] = max(24, int(c["clusters"] * 0.7))
    return c


# ---- inputs --------------------------------------------------------------------------------

def sizes_of(law, clusters, lo, hi, salt=0):
    rng = np.random.default_rng([clusters, lo, hi, salt])
    if law == "uniform":
        return rng.integers(lo, hi + 1, size=clusters)
    s = np.floor(np.exp(rng.uniform(math.log(lo), math.log(hi + 1), size=clusters))).astype(np.int64)
    return np.clip(s, lo, hi)


def pairs(c):
    return int(sizes_of(c["law"], c["clusters"], c["lo"], c["hi"]).sum()) * c["trials"]


def generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def make_points(sizes, dim, outliers, sigma, band, seed):
    """A frame's point arrays on the GPU: FP32 azimuth, elevation (3D), Doppler and int32 offsets."""
    g = generator(seed)
    sizes = np.random.default_rng(seed).permutation(sizes)
    n = torch.from_numpy(sizes).cuda()
    off = torch.zeros(len(sizes) + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(n, 0)
    npts = int(sizes.sum())
    cid = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), n)

    def u(count, a=0.0, b=1.0):
        return a + (b - a) * torch.rand(count, generator=g, device="cuda", dtype=torch.float64)

    speed, head = u(len(sizes), 0.0, 40.0), u(len(sizes), 0.0, 2.0 * math.pi)
    vx, vy = speed * torch.cos(head), speed * torch.sin(head)
    vz = u(len(sizes), -5.0, 5.0) if dim == 3 else torch.zeros_like(vx)
    az = u(npts, -60.0 * DEG, 60.0 * DEG).float()
    el = u(npts, -15.0 * DEG, 15.0 * DEG).float() if dim == 3 else None
    t, e = az.double(), 0.0 if el is None else el.double()
    ce, se = (torch.cos(e), torch.sin(e)) if dim == 3 else (1.0, 0.0)
    model = vx[cid] * torch.cos(t) * ce + vy[cid] * torch.sin(t) * ce + vz[cid] * se
    dop = model + sigma * torch.randn(npts, generator=g, device="cuda", dtype=torch.float64)

    def rank(key):  # of each point's key within its cluster
        order = torch.argsort(cid.double() * 4.0 + key)
        r = torch.empty_like(order)
        r[order] = torch.arange(npts, device="cuda") - off[cid[order]]
        return r

    n_out = torch.round(outliers * n.double()).long()
    out = rank(u(npts)) < n_out[cid]
    total = torch.sqrt(vx * vx + vy * vy + vz * vz)
    dop = torch.where(out, u(npts) * 2.0 * total[cid], dop)
    if band > 0:  # inliers moved next to the threshold
        n_band = torch.round(band * (n - n_out).double()).long()
        near = (rank(u(npts) + 2.0 * out.double()) < n_band[cid]) & ~out
        sign = torch.where(u(npts) < 0.5, -1.0, 1.0)
        dop = torch.where(near, model + sign * (TAU + u(npts, -2e-5, 2e-5)), dop)
    return az, el, dop.float(), off.int()


def make_scene(c, seed):
    """An unclustered point cloud in random order: Gaussian blobs around cells of the field of view, plus
    3% clutter.  FP32 (x, y) features, azimuth and Doppler."""
    g = generator(seed)
    gx, gy = np.meshgrid(np.arange(0.0, c["range"], 10.0) + 5.0, np.arange(-c["range"], c["range"], 10.0) + 5.0,
                         indexing="ij")
    r, a = np.hypot(gx, gy), np.arctan2(gy, gx)
    ok = (r >= 15.0) & (r <= c["range"]) & (np.abs(a) <= 60.0 * DEG)
    pick = np.random.default_rng(seed).permutation(int(ok.sum()))[:c["objects"]]
    centre = torch.from_numpy(np.stack([gx[ok][pick], gy[ok][pick]], 1)).cuda()

    def u(count, a=0.0, b=1.0):
        return a + (b - a) * torch.rand(count, generator=g, device="cuda", dtype=torch.float64)

    n_obj = c["objects"]
    centre = centre + torch.stack([u(n_obj, -1.0, 1.0), u(n_obj, -1.0, 1.0)], 1)
    sizes = torch.from_numpy(scene_sizes(c)).cuda()
    oid = torch.repeat_interleave(torch.arange(n_obj, device="cuda"), sizes)
    n_pts = oid.shape[0]
    spread = u(n_obj, 0.3, 1.2)
    xy = centre[oid] + spread[oid, None] * torch.randn(n_pts, 2, generator=g, device="cuda", dtype=torch.float64)
    speed, head = u(n_obj, 0.0, 40.0), u(n_obj, 0.0, 2.0 * math.pi)
    vx, vy = speed * torch.cos(head), speed * torch.sin(head)
    t = torch.atan2(xy[:, 1], xy[:, 0])
    dop = (vx[oid] * torch.cos(t) + vy[oid] * torch.sin(t)
           + 0.05 * torch.randn(n_pts, generator=g, device="cuda", dtype=torch.float64))
    dop = torch.where(u(n_pts) < 0.2, u(n_pts, 0.0, 2.0) * speed[oid], dop)
    n_cl = scene_points(c) - n_pts
    rr, aa = torch.exp(u(n_cl, math.log(5.0), math.log(c["range"]))), u(n_cl, -60.0 * DEG, 60.0 * DEG)
    xy = torch.cat([xy, torch.stack([rr * torch.cos(aa), rr * torch.sin(aa)], 1)])
    dop = torch.cat([dop, u(n_cl, -40.0, 40.0)])
    perm = torch.randperm(xy.shape[0], generator=g, device="cuda")
    xy = xy[perm].float().contiguous()
    az = torch.atan2(xy[:, 1].double(), xy[:, 0].double()).float()
    return xy, az, dop[perm].float().contiguous()


def scene_sizes(c):
    return sizes_of("loguniform", c["objects"], c["lo"], c["hi"], salt=1)


def scene_points(c):
    n = int(scene_sizes(c).sum())
    return n + int(round(0.03 * n))


def serving_frames(c):
    """(dim, trials, sizes, outliers, sigma) of each frame of a serving case."""
    for k in range(c["frames"]):
        dim = 2 + (k & 1)
        yield (dim, c["trials2d"] if dim == 2 else c["trials3d"],
               sizes_of("loguniform", c["clusters"], c["lo"], c["hi"], salt=2 + k), 0.20 if dim == 2 else 0.25, 0.05)


# ---- what a program keeps: a context and a stream ------------------------------------------------

_kept = {}


def kept(what):
    """The process's context for estimates and scenes, the one for serving, and its stream."""
    if what not in _kept:
        _kept[what] = torch.cuda.Stream() if what == "stream" else rvh.Context(0)
    return _kept[what]


def zero_outputs(n_clusters, n_points, device="cuda", threshold=False):
    outs = rvh.alloc_outputs(n_clusters, n_points, device, threshold=threshold)
    for t in outs.values():
        t.zero_()
    return outs


def prepare(case, seed):
    state = {"case": case, "stream": kept("stream")}
    if case["entry"] == "estimate":
        sizes = sizes_of(case["law"], case["clusters"], case["lo"], case["hi"])
        az, el, dop, off = make_points(sizes, case["dim"], case["outliers"], case["sigma"], case["band"], seed)
        outs = zero_outputs(case["clusters"], int(sizes.sum()), "cuda", threshold=case["line"])
        if case["memory"] != "device":
            def host(t):
                return None if t is None else (t.cpu().pin_memory() if case["memory"] == "pinned" else t.cpu())
            az, el, dop, off = host(az), host(el), host(dop), host(off)
            outs = {k: host(v) for k, v in outs.items()}
        state |= {"ctx": kept("context"), "inputs": (az, el, dop, off), "outs": outs,
                  "frame": rvh.make_frame(az, dop, off, el),
                  "params": rvh.make_params(case["dim"], case["trials"], TAU, seed,
                                            refine_iterations=case["refine"], confidence=case["confidence"],
                                            hypothesis_model=rvh.RVH_MODEL_PAPER_LINE if case["line"] else 0),
                  "result": rvh.make_result(outs)}
    elif case["entry"] == "scene":
        xy, az, dop = make_scene(case, seed)
        n = xy.shape[0]
        ints = {k: torch.zeros(m, dtype=torch.int32, device="cuda")
                for k, m in (("labels", n), ("perm", n), ("offsets", n + 1))}
        state |= {"ctx": kept("context"), "xy": xy, "az": az, "dop": dop, "ints": ints,
                  "gathered": (torch.zeros_like(az), torch.zeros_like(dop)),
                  "outs": zero_outputs(n, n), "params": rvh.make_params(2, case["trials"], TAU, seed)}
    else:
        frames, total_c, total_p = [], 0, 0
        for k, (dim, trials, sizes, outliers, sigma) in enumerate(serving_frames(case)):
            pts = make_points(sizes, dim, outliers, sigma, 0.0, seed * 64 + k)
            frames.append((pts, dim, trials, total_c, total_p, len(sizes), int(sizes.sum())))
            total_c, total_p = total_c + len(sizes), total_p + int(sizes.sum())
        outs = zero_outputs(total_c, total_p)
        requests = []
        for k, ((az, el, dop, off), dim, trials, c0, p0, nc, npts) in enumerate(frames):
            mine = {key: v[p0:p0 + npts] if key == "inlier_mask" else v[c0:c0 + nc] for key, v in outs.items()}
            requests.append((rvh.make_frame(az, dop, off, el), rvh.make_params(dim, trials, TAU, seed * 64 + k),
                             rvh.make_result(mine), ctypes.c_uint64(0)))
        state |= {"ctx": kept("serving"), "frames": frames, "outs": outs, "requests": requests}
    torch.cuda.synchronize()
    return state


def run(state):
    entry, ctx, stream = state["case"]["entry"], state["ctx"], state["stream"]
    if entry == "estimate":
        ctx.check(rvh.rvh_estimate(ctx.handle, state["frame"], state["params"], state["result"], stream.cuda_stream),
                  "rvh_estimate")
        return state["outs"]
    if entry == "scene":
        xy, ints, (g_az, g_dop), outs = state["xy"], state["ints"], state["gathered"], state["outs"]
        n, found = xy.shape[0], ctypes.c_int32(0)
        ctx.check(rvh.rvh_cluster(ctx.handle, xy, n, 2, EPS, MIN_PTS, ints["labels"], ints["perm"], ints["offsets"],
                                  n, found, stream.cuda_stream), "rvh_cluster")
        with torch.cuda.stream(stream):
            m = int(ints["offsets"][found.value])  # clustered points: sizes the frame
        ctx.check(rvh.rvh_gather(ctx.handle, ints["perm"], m, state["az"], g_az, state["dop"], g_dop,
                                 stream=stream.cuda_stream), "rvh_gather")
        ctx.check(rvh.rvh_estimate(ctx.handle, rvh.make_frame(g_az[:m], g_dop[:m], ints["offsets"][:found.value + 1]),
                                   state["params"], rvh.make_result(outs), stream.cuda_stream), "rvh_estimate")
        return {"clustering": ints, "gathered": [g_az, g_dop], "estimate": outs}
    for frame, params, result, ticket in state["requests"]:
        ctx.check(rvh.rvh_submit(ctx.handle, frame, params, result, ticket), "rvh_submit")
    for _, _, _, ticket in state["requests"]:
        ctx.check(rvh.rvh_wait(ctx.handle, ticket.value, -1), "rvh_wait")
    return state["outs"]


# ---- the work of one pass ------------------------------------------------------------------------

def work(case):
    """Each input read and each output written once; per (trial, point) pair the residual, k fused
    multiply-adds.  The adaptive count needs at least its first block of 128 trials."""
    def frame(n_clusters, n_points, dim, trials):
        return (n_points * (4 * dim + 1) + n_clusters * 48 + 4, 2.0 * dim * n_points * trials)

    if case["entry"] == "estimate":
        n_points = int(sizes_of(case["law"], case["clusters"], case["lo"], case["hi"]).sum())
        trials = min(case["trials"], 128) if case["confidence"] > 0 else case["trials"]
        b, f = frame(case["clusters"], n_points, case["dim"], trials)
    elif case["entry"] == "scene":
        n = scene_points(case)
        b, f = frame(case["objects"], n, 2, case["trials"])
        # features in, labels and perm out, two arrays gathered; at least one test per point
        b, f = b + n * (8 + 4 + 4 + 16), f + 5.0 * n
    else:
        parts = [frame(len(s), int(s.sum()), d, h) for d, h, s, _, _ in serving_frames(case)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    return {"bytes": float(b), "flops": float(f)}


# ---- the same results in plain FP64 torch --------------------------------------------------------

MASK32 = 0xFFFFFFFF


def philox(h, cluster, seed):
    """Philox4x32-10 of counter (h, cluster, 0, 0) under key seed: its first three words, as int64."""
    def mul(a, x):
        low, high = x & 0xFFFF, x >> 16
        return ((a * high + ((a * low) >> 16)) >> 16) & MASK32, (a * x) & MASK32

    k0, k1 = seed & MASK32, (seed >> 32) & MASK32
    x = [h, cluster, torch.zeros_like(h), torch.zeros_like(h)]
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & MASK32, (k1 + 0xBB67AE85) & MASK32
        hi0, lo0 = mul(0xD2511F53, x[0])
        hi1, lo1 = mul(0xCD9E8D57, x[2])
        x = [hi1 ^ x[1] ^ k0, lo1, hi0 ^ x[3] ^ k1, lo0]
    return x[:3]


def draw_sets(cluster, n, trials, dim, seed):
    """[B, H, dim] distinct point indices of every trial (multiply-shift with skips)."""
    h = torch.arange(trials, device="cuda")[None, :].expand(len(cluster), -1).contiguous()
    w = philox(h, cluster[:, None].expand_as(h).contiguous(), seed)
    n = n[:, None]
    q0 = (w[0] * n) >> 32
    q1 = (w[1] * (n - 1)) >> 32
    q1 = q1 + (q1 >= q0)
    if dim == 2:
        return torch.stack([q0, q1], -1)
    q2 = (w[2] * (n - 2)) >> 32
    q2 = q2 + (q2 >= torch.minimum(q0, q1))
    q2 = q2 + (q2 >= torch.maximum(q0, q1))
    return torch.stack([q0, q1, q2], -1)


def det(m):
    if m.shape[-1] == 2:
        return m[..., 0, 0] * m[..., 1, 1] - m[..., 0, 1] * m[..., 1, 0]
    return (m[..., 0, 0] * (m[..., 1, 1] * m[..., 2, 2] - m[..., 1, 2] * m[..., 2, 1])
            - m[..., 0, 1] * (m[..., 1, 0] * m[..., 2, 2] - m[..., 1, 2] * m[..., 2, 0])
            + m[..., 0, 2] * (m[..., 1, 0] * m[..., 2, 1] - m[..., 1, 1] * m[..., 2, 0]))


def cramer(m, b):
    d = det(m)
    cols = []
    for k in range(m.shape[-1]):
        mk = m.clone()
        mk[..., k] = b
        cols.append(det(mk) / d)
    return torch.stack(cols, -1), d


def least_squares(rows, w, inl, fallback):
    """Normal equations over the inliers, per cluster; fallback where they are singular."""
    k = rows.shape[-1]
    a = rows * inl[..., None]
    gram, rhs = a.transpose(1, 2) @ rows, (a.transpose(1, 2) @ w[..., None])[..., 0]
    v, d = cramer(gram, rhs)
    trace = torch.diagonal(gram, dim1=1, dim2=2).sum(-1)
    ok = (inl.sum(-1) >= k) & (d.abs() > 1e-12 * trace ** k)
    return torch.where(ok[:, None], v, fallback), ok


def median(x, valid, n):
    s = torch.where(valid, x, math.inf).sort(-1).values
    at = torch.stack([(n - 1) // 2, n // 2], -1)
    return s.gather(-1, at).mean(-1)


def exact_block(az, el, dop, start, n, cluster, dim, trials, seed, refine, confidence, line):
    """Velocities (and thresholds) of a block of clusters, padded to the largest."""
    width = int(n.max())
    j = torch.arange(width, device="cuda")[None, :]
    valid = j < n[:, None]
    at = torch.where(valid, start[:, None] + j, start[:, None])
    t, w = az[at].double(), dop[at].double()
    if dim == 3:
        e = el[at].double()
        rows = torch.stack([torch.cos(t) * torch.cos(e), torch.sin(t) * torch.cos(e), torch.sin(e)], -1)
    else:
        rows = torch.stack([torch.cos(t), torch.sin(t)], -1)
    q = draw_sets(cluster, n, trials, dim, seed)
    flat = q.flatten(1)
    thr = None
    if line:
        def unit(x):
            lo = torch.where(valid, x, math.inf).amin(-1, keepdim=True)
            hi = torch.where(valid, x, -math.inf).amax(-1, keepdim=True)
            return torch.where(hi > lo, (x - lo) / (hi - lo), torch.zeros_like(x))
        x, y = unit(t), unit(w)
        thr = median((y - median(y, valid, n)[:, None]).abs(), valid, n)
        xs, ys = x.gather(1, flat).view(q.shape), y.gather(1, flat).view(q.shape)
        dx = xs[..., 1] - xs[..., 0]
        usable = dx != 0.0
        m = (ys[..., 1] - ys[..., 0]) / torch.where(usable, dx, 1.0)
        c = ys[..., 0] - m * xs[..., 0]
        scale = torch.sqrt(m * m + 1.0)
        dist = y[:, None, :] - m[..., None] * x[:, None, :] - c[..., None]
        hits = (dist.abs() / scale[..., None] <= thr[:, None, None]) & valid[:, None, :]
        v = None
    else:
        seeds = rows.gather(1, flat[..., None].expand(-1, -1, dim)).view(*q.shape, dim)
        v, d = cramer(seeds, w.gather(1, flat).view(q.shape))
        usable = d.abs() >= (1e-4 if dim == 2 else 1e-6)
        hits = ((w[:, None, :] - v @ rows.transpose(1, 2)).abs() <= TAU) & valid[:, None, :]
    counts = torch.where(usable, hits.sum(-1), -1)
    if confidence > 0:  # trials beyond the first block after which the bound is met do not run
        best = torch.cummax(counts, 1).values
        ends = torch.arange(128, trials, 128, device="cuda")
        share = best[:, ends - 1].clamp_min(0).double() / n[:, None]
        met = ((1.0 - share ** dim) ** ends.double() <= 1.0 - confidence) & (best[:, ends - 1] >= 0)
        stop = torch.where(met.any(1), ends[met.int().argmax(1)] if len(ends) else trials,
                           torch.full_like(n, trials))
        counts = torch.where(torch.arange(trials, device="cuda")[None, :] < stop[:, None], counts, -1)
    win = (counts * trials + (trials - 1 - torch.arange(trials, device="cuda"))).argmax(1)
    inl = hits.gather(1, win[:, None, None].expand(-1, 1, width))[:, 0].double()
    nan = torch.full((len(n), dim), math.nan, dtype=torch.float64, device="cuda")
    first = nan if line else v.gather(1, win[:, None, None].expand(-1, 1, dim))[:, 0]
    out, ok = least_squares(rows, w, inl, first)
    for _ in range(refine):
        inl2 = (((w - (rows @ out[..., None])[..., 0]).abs() <= TAU) & valid).double()
        out2, ok2 = least_squares(rows, w, inl2, out)
        ok = ok & ok2
        out = torch.where(ok[:, None], out2, out)
    lost = (counts.amax(1) < 0) | (n < dim)
    return torch.where(lost[:, None], nan, out), thr


def exact_frame(az, el, dop, off, dim, trials, seed, refine=0, confidence=0.0, line=False):
    off = off.long()
    n = off[1:] - off[:-1]
    order = torch.argsort(n)
    v = torch.empty(len(n), dim, dtype=torch.float64, device="cuda")
    thr = torch.empty(len(n), dtype=torch.float64, device="cuda")
    sizes = n[order].cpu().numpy()
    a = 0
    while a < len(sizes):
        b = a + 1
        while b < len(sizes) and (b + 1 - a) * trials * int(sizes[b]) <= 1 << 28:
            b += 1
        ids = order[a:b]
        v[ids], t = exact_block(az, el, dop, off[:-1][ids], n[ids], ids, dim, trials, seed, refine, confidence, line)
        if t is not None:
            thr[ids] = t
        a = b
    out = {"vx": v[:, 0], "vy": v[:, 1], "vz": v[:, 2] if dim == 3 else torch.where(v[:, 0].isnan() & (not line),
                                                                                  math.nan, 0.0),
           "heading": torch.atan2(v[:, 1], v[:, 0])} | {k: None for k in COUNTERS}
    return out | {"threshold": thr} if line else out


def exact_dbscan(xy):
    """Labels of the scene's DBSCAN: brute-force FP64 distances, components by minimum labels."""
    p = xy.double()
    n = p.shape[0]
    src, dst = [], []
    for a in range(0, n, 2048):
        d2 = ((p[a:a + 2048, None, :] - p[None, :, :]) ** 2).sum(-1)
        i, j = (d2 <= EPS * EPS).nonzero(as_tuple=True)
        src.append((i + a).int())
        dst.append(j.int())
    src, dst = torch.cat(src).long(), torch.cat(dst).long()
    core = torch.bincount(src, minlength=n) >= MIN_PTS
    both = core[src] & core[dst]
    s, d = src[both], dst[both]
    root = torch.arange(n, device="cuda")
    while True:
        new = root.scatter_reduce(0, s, root[d], "amin")
        new = new[new]
        if torch.equal(new, root):
            break
        root = new
    # border points join their lowest-index core neighbour
    edge = ~core[src] & core[dst]
    near = torch.full((n,), n, dtype=torch.int64, device="cuda").scatter_reduce(0, src[edge], dst[edge], "amin")
    joined = ~core & (near < n)
    root = torch.where(core, root, torch.where(joined, root[near.clamp_max(n - 1)], -1))
    number = torch.cumsum((core & (root == torch.arange(n, device="cuda"))).long(), 0) - 1
    return torch.where(root >= 0, number[root.clamp_min(0)], -1)


def exact(case, seed):
    if case["entry"] == "estimate":
        sizes = sizes_of(case["law"], case["clusters"], case["lo"], case["hi"])
        az, el, dop, off = make_points(sizes, case["dim"], case["outliers"], case["sigma"], case["band"], seed)
        return exact_frame(az, el, dop, off, case["dim"], case["trials"], seed, case["refine"], case["confidence"],
                           case["line"])
    if case["entry"] == "scene":
        xy, az, dop = make_scene(case, seed)
        label = exact_dbscan(xy)
        n, count = xy.shape[0], int(label.max()) + 1
        perm = torch.argsort(torch.where(label >= 0, label, count), stable=True)[:int((label >= 0).sum())]
        off = torch.zeros(count + 1, dtype=torch.int64, device="cuda")
        off[1:] = torch.cumsum(torch.bincount(label[perm], minlength=count), 0)
        out = exact_frame(az[perm], None, dop[perm], off, 2, case["trials"], seed)
        whole = {k: None if v is None else torch.cat([v, torch.zeros(n - count, dtype=v.dtype, device="cuda")])
                 for k, v in out.items()}
        rest = torch.zeros(n - len(perm), dtype=torch.float64, device="cuda")
        return {"clustering": {"labels": None, "perm": None, "offsets": None},
                "gathered": [torch.cat([x[perm].double(), rest]) for x in (az, dop)], "estimate": whole}
    parts = []
    for k, (dim, trials, sizes, outliers, sigma) in enumerate(serving_frames(case)):
        az, el, dop, off = make_points(sizes, dim, outliers, sigma, 0.0, seed * 64 + k)
        parts.append(exact_frame(az, el, dop, off, dim, trials, seed * 64 + k))
    return {k: None if v is None else torch.cat([p[k] for p in parts]) for k, v in parts[0].items()}
