"""Performance cases: the work that a user of this library has it do.

Every case is one call sequence through the public binding
(``paper_2311_17604_gb300.pd``) on a synthetic terrestrial-LiDAR scan.  The
scans are those of the library's own workloads (a box room, an outdoor scene,
a merged multi-station site), cast here on the GPU so that fresh inputs cost
little: rays on a uniform azimuth x elevation grid, 2 mm range noise, int32
millimetres.

    listed()             the cases that are reported
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  inputs on the GPU (host arrays for the served scans)
    run(state)           one pass; returns every output
    work(case)           bytes and flops that a pass cannot do without
    exact(case, seed)    the floating outputs in 64 bits, where that is quick

Kinds of cases:
    static    pd_knn_cost_static: the allocation-free pass of a real-time
              ingest loop on one small packet of a scan (latency)
    knn       pd_build_grid + pd_knn_cost: costs and neighbours of a cloud
    decimate  pd_build_grid + pd_decimate_ratio (density cost): the library's
              main use, from a room scan to a merged site
    wup       pd_build_grid + pd_decimate_wup: the paper's iterative scheme
    batch     pd_decimate_batch, packed: many room scans, colour term
    serve     Server.submit / poll: host scans in, keep masks out, normals by
              the network, orientation term
    normals   pd_build_grid + pd_normals_pca + pd_normals_mlp
    forward   pd_mlp_forward: network inference alone
    train     MlpTrainer.train: Adam steps of the normals network
    quality   pd_quality_report of a decimated cloud
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2311_17604_gb300.pd as pd

KNN_OF_NORMALS = 16
ROW = 48          # features of a row
HIDDEN = 64
OUTDOOR_RETURNS = 0.49  # share of the outdoor scene's rays that give a point (rest: sky, dropout)


# ------------------------------------------------------------------ cases
def listed():
    return [
        # one sweep packet of a moving scanner: the smallest call, launch latency
        {"name": "static_7k_k4", "kind": "static", "n_az": 145, "n_el": 51, "k": 4},
        # costs and neighbours of an ordinary room scan
        {"name": "knn_room_1m_k6", "kind": "knn", "scene": "room", "stations": 1,
         "n_az": 2260, "n_el": 451, "k": 6},
        # the 200k-point room scan, k = 1, keep 25 %: an interactive call
        {"name": "room_200k_k1", "kind": "decimate", "scene": "room", "stations": 1,
         "n_az": 1000, "n_el": 200, "k": 1, "ratio": 0.25},
        # the 20M-ray outdoor scan, k = 4, keep 10 %
        {"name": "outdoor_10m_k4", "kind": "decimate", "scene": "outdoor", "stations": 1,
         "n_az": 10000, "n_el": 2000, "k": 4, "ratio": 0.10},
        # four merged stations of the site scan, k = 1, keep 5 %: the largest
        {"name": "site_100m_k1", "kind": "decimate", "scene": "site", "stations": 4,
         "n_az": 10000, "n_el": 2500, "k": 1, "ratio": 0.05},
        # the paper's own scheme on a room scan, with its k = 6
        {"name": "wup_room_700k_k6", "kind": "wup", "scene": "room", "stations": 1,
         "n_az": 1871, "n_el": 374, "k": 6, "ratio": 0.20},
        # a batch of uneven room scans with the 0.3 colour term
        {"name": "batch_12_colour", "kind": "batch", "scans": 12, "lo": 50000, "hi": 1000000,
         "k": 1, "weight": 0.3},
        # served room scans: network normals, k = 4 + 0.5 x orientation, keep 25 %
        {"name": "serve_4_orient", "kind": "serve", "scans": 4, "lo": 100000, "hi": 1000000,
         "k": 4, "weight": 0.5, "ratio": 0.25},
        # normals of a whole room scan: 16 nearest, PCA, network
        {"name": "normals_room_2m", "kind": "normals", "scene": "room", "stations": 1,
         "n_az": 3163, "n_el": 633},
        # inference over the rows of a large scan
        {"name": "forward_4m_rows", "kind": "forward", "rows": 4000003},
        # one training call: 200 Adam steps of 4096 rows
        {"name": "train_200x4096", "kind": "train", "rows": 300000, "steps": 200, "batch": 4096},
        # quality of a decimated room scan, radii from 2 to 20 cm
        {"name": "quality_room_1m", "kind": "quality", "scene": "room", "stations": 1,
         "n_az": 2240, "n_el": 447, "keep": 0.25, "radii": 7, "r_max": 200},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid_of(rng, n):
    """Azimuth and elevation steps of about n rays, about 5 : 1, any remainder."""
    n_el = max(8, int(round(math.sqrt(n / rng.uniform(4.0, 6.0)))))
    return max(8, int(round(n / n_el))), n_el


def draw(rng):
    kind = rng.choice(["static", "knn", "decimate", "decimate", "decimate", "wup", "batch",
                       "serve", "normals", "forward", "train", "quality"])
    if kind == "static":
        n_az, n_el = _grid_of(rng, _log(rng, 500, 60000))
        return {"kind": kind, "n_az": n_az, "n_el": n_el, "k": rng.choice([1, 4, 6, 16])}
    if kind == "knn":
        n_az, n_el = _grid_of(rng, _log(rng, 20000, 5e6))
        return {"kind": kind, "scene": rng.choice(["room", "site"]), "stations": 1,
                "n_az": n_az, "n_el": n_el, "k": rng.choice([1, 2, 4, 6, 16])}
    if kind == "decimate":
        k = rng.choice([1, 1, 4])
        scene = rng.choice(["room", "outdoor", "site"])
        top = 8e7 if k == 1 and scene == "site" else 5e6
        st = rng.choice([1, 2, 3]) if scene == "site" else 1
        n_az, n_el = _grid_of(rng, _log(rng, 50000, top) / st)
        return {"kind": kind, "scene": scene, "stations": st, "n_az": n_az, "n_el": n_el,
                "k": k, "ratio": round(rng.uniform(0.05, 0.5), 3)}
    if kind == "wup":
        n_az, n_el = _grid_of(rng, _log(rng, 50000, 700000))
        return {"kind": kind, "scene": "room", "stations": 1, "n_az": n_az, "n_el": n_el,
                "k": rng.choice([1, 4, 6]), "ratio": round(rng.uniform(0.1, 0.5), 3)}
    if kind == "batch":
        return {"kind": kind, "scans": rng.randint(3, 12), "lo": 50000,
                "hi": int(_log(rng, 100000, 900000)), "k": 1, "weight": 0.3}
    if kind == "serve":
        return {"kind": kind, "scans": rng.randint(1, 4), "lo": 100000,
                "hi": int(_log(rng, 150000, 900000)), "k": 4, "weight": 0.5, "ratio": 0.25}
    if kind == "normals":
        n_az, n_el = _grid_of(rng, _log(rng, 100000, 3e6))
        return {"kind": kind, "scene": "room", "stations": 1, "n_az": n_az, "n_el": n_el}
    if kind == "forward":
        return {"kind": kind, "rows": int(_log(rng, 1000, 6e6))}
    if kind == "train":
        return {"kind": kind, "rows": int(_log(rng, 20000, 500000)), "steps": rng.randint(20, 250),
                "batch": int(_log(rng, 500, 8192))}
    n_az, n_el = _grid_of(rng, _log(rng, 50000, 2e6))
    return {"kind": "quality", "scene": "room", "stations": 1, "n_az": n_az, "n_el": n_el,
            "keep": round(rng.uniform(0.1, 0.4), 3), "radii": rng.randint(3, 8),
            "r_max": rng.randint(60, 200)}


# ------------------------------------------------------------------ scans
def _dev(v):
    return torch.tensor(v, dtype=torch.float32, device="cuda")


def _inside_box(o, d, lo, hi):
    """Exit distance of rays that start inside the box."""
    t = torch.where(d > 0, (hi - o) / d, (lo - o) / d)
    return torch.nan_to_num(t, nan=math.inf).amin(dim=1)


def _outside_box(o, d, lo, hi):
    """Entry distance of rays that start outside the box (inf: no hit)."""
    t1, t2 = (lo - o) / d, (hi - o) / d
    near, far = torch.minimum(t1, t2).amax(dim=1), torch.maximum(t1, t2).amin(dim=1)
    return torch.where((near <= far) & (near > 1e-6), near, math.inf)


def _sphere(o, d, c, r):
    oc = o - c
    b = d @ oc
    disc = b * b - (oc @ oc - r * r)
    t = -b - disc.clamp_min(0).sqrt()
    return torch.where((disc >= 0) & (t > 1e-6), t, math.inf)


def _cylinder(o, d, c, r, h):
    """Side of a vertical cylinder that stands on the ground."""
    ox, oy = o[0] - c[0], o[1] - c[1]
    a = d[:, 0] ** 2 + d[:, 1] ** 2
    b = ox * d[:, 0] + oy * d[:, 1]
    disc = b * b - a * (ox * ox + oy * oy - r * r)
    t = (-b - disc.clamp_min(0).sqrt()) / a
    z = o[2] + t * d[:, 2]
    return torch.where((disc >= 0) & (t > 1e-6) & (z >= 0) & (z <= h), t, math.inf)


def _scene(kind, r, stations):
    """Primitives (a distance function each) and the stations' positions."""
    u = r.uniform
    if kind == "room":
        dims = (10.0 * u(0.8, 1.2), 8.0 * u(0.8, 1.2), 3.0 * u(0.8, 1.2))
        pos = [(dims[0] * u(0.3, 0.5), dims[1] * u(0.3, 0.5), 1.5)]
        prims = [lambda o, d, hi=_dev(dims): _inside_box(o, d, 0 * hi, hi)]
        for _ in range(3):  # boxes in the far half of the room
            side = (u(0.4, 1.5), u(0.4, 1.5), u(0.4, 1.5))
            lo = (u(0.6 * dims[0], dims[0] - 1.6), u(0.0, dims[1] - 1.6), 0.0)
            hi = tuple(a + b for a, b in zip(lo, side))
            prims.append(lambda o, d, lo=_dev(lo), hi=_dev(hi): _outside_box(o, d, lo, hi))
        return prims, pos
    if kind == "outdoor":
        prims = [lambda o, d: torch.where(d[:, 2] < 0, -o[2] / d[:, 2], math.inf)]
        for i in range(60):  # 40 boxes and 20 spheres at 4 to 60 m
            dist, th = u(4.0, 60.0), u(0.0, 2 * math.pi)
            cx, cy = dist * math.cos(th), dist * math.sin(th)
            if i < 40:
                w, v, h = u(0.5, 4.0), u(0.5, 4.0), u(0.5, 12.0)
                lo, hi = (cx - w / 2, cy - v / 2, 0.0), (cx + w / 2, cy + v / 2, h)
                prims.append(lambda o, d, lo=_dev(lo), hi=_dev(hi): _outside_box(o, d, lo, hi))
            else:
                rad = u(0.3, 2.5)
                prims.append(lambda o, d, c=_dev((cx, cy, rad)), rad=rad: _sphere(o, d, c, rad))
        return prims, [(0.0, 0.0, 1.5)]
    # site: a closed 200 x 200 x 30 m shell, 30 boxes and 30 cylinders, the
    # stations along a free lane in the middle
    prims = [lambda o, d, hi=_dev((200.0, 200.0, 30.0)): _inside_box(o, d, 0 * hi, hi)]
    for i in range(60):
        y0 = u(2.0, 65.0) if i % 2 else u(110.0, 170.0)
        x0 = u(2.0, 170.0)
        if i < 30:
            lo, hi = (x0, y0, 0.0), (x0 + u(2.0, 25.0), y0 + u(2.0, 25.0), u(2.0, 20.0))
            prims.append(lambda o, d, lo=_dev(lo), hi=_dev(hi): _outside_box(o, d, lo, hi))
        else:
            c, rad, h = (x0 + 3, y0 + 3), u(0.15, 3.0), u(2.0, 25.0)
            prims.append(lambda o, d, c=c, rad=rad, h=h: _cylinder(o, d, c, rad, h))
    return prims, [(u(5.0, 195.0), u(95.0, 105.0), 1.5) for _ in range(stations)]


def scan(kind, seed, stations, n_az, n_el, colours=False):
    """Merged scan of `stations` stations: int32 [n, 3] mm on the GPU (and uint8
    [n, 3] colours).  Points are in acquisition order (azimuth, then elevation)."""
    r = random.Random("%s %d" % (kind, seed))
    prims, pos = _scene(kind, r, stations)
    base = torch.tensor([[r.randint(40, 255) for _ in range(3)] for _ in prims],
                        dtype=torch.float32, device="cuda")
    gen = torch.Generator(device="cuda").manual_seed(seed)
    xyz, rgb = [], []
    el = (torch.arange(n_el, device="cuda") + 0.5) * (math.pi / n_el) - 0.5 * math.pi
    step = max(1, (1 << 23) // n_el)
    for p in pos:
        o = _dev(p)
        for a0 in range(0, n_az, step):
            az = torch.arange(a0, min(n_az, a0 + step), device="cuda") * (2 * math.pi / n_az)
            d = torch.empty(len(az), n_el, 3, device="cuda")
            d[..., 0] = az.cos()[:, None] * el.cos()
            d[..., 1] = az.sin()[:, None] * el.cos()
            d[..., 2] = el.sin()
            d = d.reshape(-1, 3)
            d = torch.where(d == 0, 1e-9, d)  # no division by zero below
            t = prims[0](o, d)
            hit = torch.zeros(len(t), dtype=torch.int64, device="cuda") if colours else None
            for i, f in enumerate(prims[1:], 1):
                ti = f(o, d)
                if colours:
                    hit = torch.where(ti < t, i, hit)
                t = torch.minimum(t, ti)
            t = t + 0.002 * torch.randn(len(t), device="cuda", generator=gen)
            q = o + t[:, None] * d
            if kind == "outdoor":
                q = torch.where((t < 120.0)[:, None], q, math.nan)  # sky: no return
            xyz.append((q * 1000.0 + 0.5).floor())
            if colours:
                odd = (q / 0.5).floor().to(torch.int64).sum(dim=1) & 1
                rgb.append((base[hit] * torch.where(odd == 0, 1.0, 0.6)[:, None]).to(torch.uint8))
    xyz = torch.cat(xyz)
    if kind == "outdoor":  # returns within 120 m, all but a fixed number of them dropped
        at = (~xyz[:, 0].isnan()).nonzero()[:, 0]
        at = at[torch.randperm(len(at), device="cuda", generator=gen)]
        xyz = xyz[at[:int(n_az * n_el * OUTDOOR_RETURNS)].sort().values]
    xyz = xyz.to(torch.int32).contiguous()
    return (xyz, torch.cat(rgb).contiguous()) if colours else xyz


def _scan_sizes(case):
    """Rays per scan of a batch: spread over the logarithm of the range."""
    c = case["scans"]
    out = []
    for i in range(c):
        n = case["lo"] * (case["hi"] / case["lo"]) ** ((i + 0.5) / c)
        n_el = max(8, int(round(math.sqrt(n / 5.0))))
        out.append((5 * n_el + i, n_el))
    return out


# ------------------------------------------------------------------ network rows
def _rows(n, seed):
    """Feature rows (bfloat16 bits, int16 [n, 48]) of noisy planar neighbourhoods
    and their unit normals (float32 [n, 3])."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    feat = torch.empty(n, ROW, dtype=torch.int16, device="cuda")
    labels = torch.empty(n, 3, dtype=torch.float32, device="cuda")
    for b in range(0, n, 1 << 20):
        m = min(n, b + (1 << 20)) - b
        f = torch.randn(m, 3, 3, device="cuda", generator=gen)
        w = f[:, 0] / f[:, 0].norm(dim=1, keepdim=True)
        u = torch.linalg.cross(w, f[:, 1])
        u = u / u.norm(dim=1, keepdim=True)
        v = torch.linalg.cross(w, u)
        r = torch.rand(m, KNN_OF_NORMALS, device="cuda", generator=gen).sqrt().sort(dim=1).values
        th = torch.rand(m, KNN_OF_NORMALS, device="cuda", generator=gen) * (2 * math.pi)
        h = 0.1 * torch.randn(m, KNN_OF_NORMALS, device="cuda", generator=gen)
        x = ((r * th.cos())[..., None] * u[:, None] + (r * th.sin())[..., None] * v[:, None]
             + h[..., None] * w[:, None])
        x = x / x.square().sum(dim=2).mean(dim=1).sqrt()[:, None, None]
        feat[b:b + m] = x.reshape(m, ROW).to(torch.bfloat16).view(torch.int16)
        labels[b:b + m] = w
    return feat, labels


def _initial(seed):
    """Untrained parameters W1 b1 W2 b2 W3 b3 in the library's flat layout."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for rows, cols, s in ((HIDDEN, ROW, 6.0), (HIDDEN, HIDDEN, 6.0), (3, HIDDEN, 3.0)):
        w = torch.rand(rows, cols, device="cuda", generator=gen) * 2 - 1
        out += [(w * math.sqrt(s / cols)).reshape(-1), torch.zeros(rows, device="cuda")]
    return torch.cat(out).contiguous()


def _unpack(p):
    o, out = 0, []
    for rows, cols in ((HIDDEN, ROW), (HIDDEN, HIDDEN), (3, HIDDEN)):
        out.append(p[o:o + rows * cols].reshape(rows, cols))
        o += rows * cols
        out.append(p[o:o + rows])
        o += rows
    return out


def _net(p, x):
    w1, b1, w2, b2, w3, b3 = _unpack(p)
    return ((x @ w1.T + b1).relu() @ w2.T + b2).relu() @ w3.T + b3


_TRAINED = None


def _trained():
    """The weights that a serving program keeps: trained once on noisy planes."""
    global _TRAINED
    if _TRAINED is None:
        feat, y = _rows(8192, 1)
        x = feat.view(torch.bfloat16).float()
        p = _initial(1).requires_grad_(True)
        opt = torch.optim.Adam([p], lr=3e-3)
        for _ in range(300):
            n = _net(p, x)
            loss = (1 - (n / n.norm(dim=1, keepdim=True) * y).sum(dim=1).square()).mean()
            opt.zero_grad()
            loss.backward()
            opt.step()
        _TRAINED = p.detach().clone()
    return _TRAINED


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "kind": kind}
    if kind == "static":
        s["xyz"] = scan("room", seed, 1, case["n_az"], case["n_el"])
    elif kind in ("knn", "decimate", "wup", "normals", "quality"):
        s["ctx"] = pd.Context()
        s["xyz"] = scan(case["scene"], seed, case["stations"], case["n_az"], case["n_el"])
        if kind == "normals":
            s["net"] = _trained()
        if kind == "quality":
            gen = torch.Generator(device="cuda").manual_seed(seed)
            u = torch.rand(len(s["xyz"]), device="cuda", generator=gen)
            s["keep"] = (u < case["keep"]).to(torch.uint8)
    elif kind == "batch":
        s["ctx"] = pd.Context()
        r = random.Random(seed)
        s["clouds"] = []
        for i, (n_az, n_el) in enumerate(_scan_sizes(case)):
            xyz, rgb = scan("room", seed * 1009 + i, 1, n_az, n_el, colours=True)
            s["clouds"].append({"xyz": xyz, "rgb": rgb, "ratio": r.uniform(0.05, 0.5)})
    elif kind == "serve":
        s["ctx"] = pd.Context()
        s["server"] = pd.Server(s["ctx"], slots=4, mem_budget=16 << 30, k=case["k"],
                                term=pd.PD_TERM_ORIENT, weight=case["weight"],
                                mlp_params=_trained(), normals=True)
        s["scans"] = []
        for i, (n_az, n_el) in enumerate(_scan_sizes(case)):
            xyz = scan("room", seed * 1009 + i, 1, n_az, n_el)
            s["scans"].append((pd.pinned_like(xyz.cpu().numpy()),
                               pd.pinned_like(np.zeros(len(xyz), dtype=np.uint8))))
    elif kind == "forward":
        s["net"] = _trained()
        s["feat"], _ = _rows(case["rows"], seed)
    elif kind == "train":
        s["ctx"] = pd.Context()
        s["feat"], s["labels"] = _rows(case["rows"], seed)
        gen = torch.Generator(device="cuda").manual_seed(seed)
        u = torch.rand(case["rows"], device="cuda", generator=gen)
        s["valid"] = (u < 0.8).to(torch.uint8)  # rows that PCA found planar
        s["initial"] = _initial(seed)
        s["seed"] = seed
    else:
        raise ValueError(kind)
    return s


# ------------------------------------------------------------------ run
def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "static":
        return pd.pd_knn_cost_static(s["xyz"], k=case["k"])
    if kind == "knn":
        g = pd.Grid(s["ctx"], s["xyz"])
        out = pd.pd_knn_cost(g, k=case["k"])
        g.free()
        return out
    if kind == "decimate":
        g = pd.Grid(s["ctx"], s["xyz"])
        keep = pd.pd_decimate_ratio(g, case["ratio"], k=case["k"])
        g.free()
        return keep
    if kind == "wup":
        g = pd.Grid(s["ctx"], s["xyz"])
        keep = pd.pd_decimate_wup(g, int(case["ratio"] * g.n), k=case["k"])
        g.free()
        return keep
    if kind == "batch":
        keeps, _ = pd.pd_decimate_batch(s["ctx"], s["clouds"], k=case["k"],
                                        term=pd.PD_TERM_COLOR, weight=case["weight"])
        return keeps
    if kind == "serve":
        srv = s["server"]
        tickets = [srv.submit(xyz, ratio=case["ratio"], keep=keep) for xyz, keep in s["scans"]]
        return [srv.poll(t)[0] for t in tickets]
    if kind == "normals":
        g = pd.Grid(s["ctx"], s["xyz"])
        feat, pca, valid = pd.pd_normals_pca(g)
        normals = pd.pd_normals_mlp(s["ctx"], s["net"], feat, pca)
        g.free()
        return feat, pca, valid, normals
    if kind == "forward":
        return pd.pd_mlp_forward(s["net"], s["feat"])
    if kind == "train":
        t = pd.MlpTrainer(params=s["initial"].clone())
        loss = t.train(s["ctx"], s["feat"], s["labels"], valid=s["valid"], steps=case["steps"],
                       batch=case["batch"], lr=1e-3, seed=s["seed"])
        return t.params, t.adam, loss
    q = pd.pd_quality_report(s["ctx"], s["xyz"], s["keep"], _radii(case))
    return {"points": q["points"], "mean": np.array(q["mean"]),
            "fractile": np.array(q["fractile"], dtype=np.int64),
            "fit": np.array([q["slope_per_m2"], q["intercept"], q["r2"], q["rmse"]]),
            "min_spacing2": q["min_spacing2_mm2"], "mean_spacing": q["mean_spacing_mm"]}


def _radii(case):
    return [int(round(case["r_max"] * (j + 1) / case["radii"])) for j in range(case["radii"])]


# ------------------------------------------------------------------ work
def _points(case):
    if "rows" in case:
        return case["rows"]
    if "scans" in case:
        return sum(a * e for a, e in _scan_sizes(case))
    n = case["n_az"] * case["n_el"] * case.get("stations", 1)
    return int(n * OUTDOOR_RETURNS) if case.get("scene") == "outdoor" else n


def work(case):
    """Each input read once and each output written once; flops of the network."""
    kind, n = case["kind"], _points(case)
    net = 2 * (ROW * HIDDEN + HIDDEN * HIDDEN + 3 * HIDDEN)  # of one row's forward
    if kind in ("static", "knn"):
        return {"bytes": n * (12 + 8 + 4 * case["k"]), "flops": 0}
    if kind in ("decimate", "wup", "serve"):
        return {"bytes": n * (12 + 1), "flops": n * net if kind == "serve" else 0}
    if kind == "batch":
        return {"bytes": n * (12 + 3 + 1), "flops": 0}
    if kind == "normals":
        return {"bytes": n * (12 + 2 * ROW + 12 + 1 + 12), "flops": n * net}
    if kind == "forward":
        return {"bytes": n * (2 * ROW + 12 + 4), "flops": n * net}
    if kind == "train":
        rows = case["steps"] * case["batch"]
        return {"bytes": rows * (2 * ROW + 12), "flops": rows * 3 * net}
    return {"bytes": n + n * case["keep"] * 12, "flops": 0}


# ------------------------------------------------------------------ exact
MOST_PAIRS = 5e10  # brute force over all pairs, a few seconds


def _nearest(x, k):
    """Ascending squared distances to the k nearest others (float64, exact)."""
    x = x.to(torch.float64)
    out = []
    step = max(1, (1 << 28) // len(x))
    for b in range(0, len(x), step):
        d = torch.zeros(min(len(x), b + step) - b, len(x), dtype=torch.float64, device="cuda")
        for a in range(3):
            d += (x[b:b + step, a:a + 1] - x[None, :, a]).square()
        d[torch.arange(len(d)), torch.arange(b, b + len(d))] = math.inf
        out.append(d.topk(k, dim=1, largest=False).values)
    return torch.cat(out)


def exact(case, seed):
    kind, n = case["kind"], _points(case)
    if kind in ("static", "knn") and n * float(n) <= MOST_PAIRS:
        x = prepare(case, seed)["xyz"]
        return (1.0 / _nearest(x, case["k"])).sum(dim=1), None
    if kind == "forward":
        s = prepare(case, seed)
        norm, unit = [], []
        for f in s["feat"].split(1 << 19):
            o = _net(s["net"].double(), f.view(torch.bfloat16).double())
            norm.append(o.norm(dim=1))
            unit.append(o / norm[-1][:, None])
        return torch.cat(unit), torch.cat(norm)
    if kind == "quality" and (n * case["keep"]) ** 2 * case["radii"] <= MOST_PAIRS:
        s = prepare(case, seed)
        x = s["xyz"][s["keep"] != 0].to(torch.float64)
        r = _radii(case)
        counts = torch.zeros(len(x), len(r), dtype=torch.float64, device="cuda")
        near = []
        step = max(1, (1 << 27) // len(x))
        for b in range(0, len(x), step):
            d = torch.zeros(min(len(x), b + step) - b, len(x), dtype=torch.float64, device="cuda")
            for a in range(3):
                d += (x[b:b + step, a:a + 1] - x[None, :, a]).square()
            d[torch.arange(len(d)), torch.arange(b, b + len(d))] = math.inf
            for j, v in enumerate(r):
                counts[b:b + step, j] = (d <= float(v * v)).sum(dim=1)
            near.append(d.amin(dim=1))
        area = torch.tensor([math.pi * (v / 1000.0) ** 2 for v in r], dtype=torch.float64,
                            device="cuda")
        dx, dy = area - area.mean(), counts - counts.mean()
        slope = float((dx * dy).sum() / (dx.square().sum() * len(x)))
        res = dy - slope * dx
        fit = np.array([slope, float(counts.mean() - slope * area.mean()),
                        1.0 - float(res.square().sum() / dy.square().sum()),
                        math.sqrt(float(res.square().mean()))])
        return {"points": None, "mean": counts.mean(dim=0).cpu().numpy(), "fractile": None,
                "fit": fit, "min_spacing2": None,
                "mean_spacing": float(torch.cat(near).sqrt().mean())}
    return None
