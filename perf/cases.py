"""The work that users of this library have it do, as timed cases.

A case is a dict of plain values.  Its ``kind`` says which public call it
stands for; the rest are the lens model, the map and the options that a user
would pass.  Sizes follow the workloads of ``bench.py`` and the tests: maps
from tens to thousands of pixels a side with 20 to 100 rays landing per pixel,
star fields from about a hundred to a hundred thousand stars, equal, Salpeter
(0.1-1) and Kroupa (0.08-1.5) masses, expansion orders 20 to 40.

    listed()             the cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  what a program holds before the call
    run(state)           one pass through the public entry points
    work(case)           bytes and flops that one pass cannot do without
    exact(case, seed)    the same outputs in 64 bits by a direct sum over the
                         stars, for cases small enough
"""
import math
import random

import numpy as np
import torch

import paper_2506_02114_gb300 as mm

# piecewise power laws dN/dm ~ m^-alpha: segment edges and exponents
MASSES = {"equal": None,
          "salpeter": ((0.1, 1.0), (2.35,)),
          "kroupa": ((0.08, 0.5, 1.5), (1.3, 2.3))}

MAX_RAYS = 6.6e9        # grid rays of the largest listed map
MAX_LANDING = 2.5e9     # of which inside the map, without stars
MAX_PAIRS = 4.0e9       # ray-star pairs of a direct-sum map


def listed():
    return [
        # source positions of a few thousand image points (light curves, image finding): a
        # small synchronous call, host arrays in and out
        _case("points_4096", "points", 0.4, 0.3, 0.0, "equal", 4.0, 256, 20.0, f=0.01, points=4096),
        # a thumbnail map: launches and latency, not throughput
        _case("map_48", "map", 0.45, 0.3, 0.4, "equal", 1.5, 48, 38.0, f=0.01, order=20),
        # a preview of a large field: many stars, few rays, so the tree and the expansions count
        _case("map_400_50k_stars", "map", 0.5, 0.4, 0.5, "salpeter", 10.0, 400, 20.0),
        # a rectangular star region, an oblong map away from the origin
        _case("map_601x1003_rect", "map", 0.45, 0.3, 0.3, "salpeter", 6.0, 601, 100.0, npix_y=1003,
              center_x=0.7, center_y=-0.4, rect=True),
        # a map of a parameter survey, with the leaf size its tuning usually ends at
        _case("map_1237_survey", "map", 0.62, 0.21, 0.3, "salpeter", 11.3, 1237, 100.0, leaf=16,
              rows_per_item=512),
        # the benchmark's single map
        _case("map_2000", "map", 0.5, 0.4, 0.5, "salpeter", 10.0, 2000, 100.0),
        # close to the macro model's critical curve (sliver triangles), larger than L2
        _case("map_3001_near_critical", "map", 0.8, 0.25, 0.0, "equal", 6.0, 3001, 25.0, f=0.005,
              order=30),
        # the largest: high order, most of its rays inside the map
        _case("map_5000_kroupa", "map", 0.5, 0.45, 0.8, "kroupa", 12.5, 5000, 100.0, order=40),
        # rays counted per pixel instead of polygons
        _case("irs_1537", "irs", 0.5, 0.4, 0.5, "salpeter", 8.0, 1537, 100.0),
        # the direct sum in 64 bits: 160 stars, an explicit 700 x 2000 grid
        _case("plain_256", "plain", 0.4, 0.3, 0.0, "equal", 4.0, 256, 20.0, stars=160, radius=20.0,
              img_half_x=16.0 / 3.0, img_half_y=16.0, rays_x=700, rays_y=2000),
        # several maps of a survey in one call
        _case("batch_12", "batch", 0.0, 0.0, 0.0, "salpeter", 0.0, 0, 100.0, maps=12, npix_min=500,
              npix_max=1000, draw=11),
        # a new star field each time: plan, run, read back, release
        _case("one_shot_800", "one_shot", 0.6, 0.2, 0.6, "kroupa", 7.0, 800, 100.0),
    ]


def _case(name, kind, kappa, gamma, s, mass, half_length, npix, landing, f=1e-3, order=25, **more):
    c = {"name": name, "kind": kind, "kappa": kappa, "gamma": gamma, "s": s, "mass": mass,
         "half_length": half_length, "npix": npix, "landing": landing, "f": f, "order": order}
    c.update(more)
    return c


# ---------------------------------------------------------------------------
# sizes of a case
# ---------------------------------------------------------------------------

def _moment(mass, q):
    """Unnormalised integral of m^q dN/dm."""
    edges, alphas = MASSES[mass]
    tot, c = 0.0, 1.0
    for k, a in enumerate(alphas):
        if k:
            c *= edges[k] ** (a - alphas[k - 1])
        e = q + 1 - a
        tot += c * (edges[k + 1] ** e - edges[k] ** e) / e
    return tot


def _mean_mass(mass):
    return 1.0 if MASSES[mass] is None else _moment(mass, 1) / _moment(mass, 0)


def _geometry(c):
    """The shooting region, ray spacing, star region and counts of a single-map case."""
    ks = (1.0 - c["s"]) * c["kappa"]
    m2 = 1.0 if MASSES[c["mass"]] is None else _moment(c["mass"], 2) / _moment(c["mass"], 1)
    a = (1.0 - c["kappa"] + c["gamma"], 1.0 - c["kappa"] - c["gamma"])
    nx, ny = c["npix"], c.get("npix_y", 0) or c["npix"]
    delta = 2.0 * c["half_length"] / nx
    side = (c["half_length"], 0.5 * ny * delta)
    centre = (c.get("center_x", 0.0), c.get("center_y", 0.0))
    r = math.sqrt(ks * m2 / c["f"])
    rpp = c["landing"] * abs(a[0] * a[1])
    half = tuple((side[k] + r) / abs(a[k]) for k in (0, 1))
    mid = tuple(centre[k] / a[k] for k in (0, 1))
    if "rays_x" in c:
        half = (c["img_half_x"], c["img_half_y"])
        n = (c["rays_x"], c["rays_y"])
        h = tuple(2.0 * half[k] / (n[k] - 1) for k in (0, 1))
        x0 = tuple(mid[k] - half[k] for k in (0, 1))
    else:
        hh = delta / math.sqrt(rpp)
        n = tuple(int(math.ceil(2.0 * half[k] / hh)) + 1 for k in (0, 1))
        h = (hh, hh)
        x0 = tuple(mid[k] - 0.5 * (n[k] - 1) * hh for k in (0, 1))
    reach = tuple(half[k] + abs(mid[k]) for k in (0, 1))
    radius = c.get("radius", 1.1 * math.hypot(*reach))
    rect = tuple(1.1 * x + 1.0 for x in reach) if c.get("rect") else None
    per_area = ks / (math.pi * _mean_mass(c["mass"]))
    area = 4.0 * rect[0] * rect[1] if rect else math.pi * radius * radius
    stars = c.get("stars") or int(round(per_area * area))
    return {"ks": ks, "nx": nx, "ny": ny, "delta": delta, "side": side, "centre": centre,
            "half": half, "n": n, "h": h, "x0": x0, "rpp": rpp, "radius": radius, "rect": rect,
            "stars": stars, "rays": float(n[0]) * n[1], "landing": float(nx) * ny * c["landing"]}


def _survey(rng, npix_min, npix_max):
    """A survey's map: kappa in [0.2, 0.9], gamma in [0.1, 0.8] away from the critical line."""
    while True:
        kappa, gamma = rng.uniform(0.2, 0.9), rng.uniform(0.1, 0.8)
        if abs(abs(1.0 - kappa) - gamma) >= 0.05:
            break
    npix = int(round(math.exp(rng.uniform(math.log(npix_min), math.log(npix_max)))))
    return {"kappa": kappa, "gamma": gamma, "s": rng.choice((0.0, 0.3, 0.6, 0.9)), "npix": npix,
            "half_length": rng.uniform(5.0, 20.0) * min(1.0, npix / 500.0)}


def _batch_maps(c):
    """The single-map cases of a batch."""
    rng = random.Random(c["draw"])
    out = []
    while len(out) < c["maps"]:
        m = {"kind": "map", "mass": c["mass"], "landing": c["landing"], "f": c["f"],
             "order": c["order"]}
        m.update(_survey(rng, c["npix_min"], c["npix_max"]))
        g = _geometry(m)
        if 100 <= g["stars"] <= 100000 and g["rays"] <= 4e8:
            out.append(m)
    return out


def draw(rng):
    while True:
        kind = rng.choice(("map", "map", "map", "map", "irs", "irs", "plain", "batch", "one_shot",
                           "points"))
        c = {"kind": kind, "mass": rng.choice(("equal", "salpeter", "kroupa")),
             "landing": round(rng.uniform(20.0, 100.0), 1), "f": rng.choice((1e-3, 2e-3, 5e-3, 1e-2)),
             "order": rng.choice((20, 25, 25, 25, 30, 40))}
        if kind == "batch":
            lo = rng.randint(60, 500)
            c.update(kappa=0.0, gamma=0.0, s=0.0, half_length=0.0, npix=0, maps=rng.randint(2, 16),
                     npix_min=lo, npix_max=2 * lo, draw=rng.randint(0, 1 << 20))
            return c
        top = {"map": 3500, "irs": 2000, "plain": 256, "one_shot": 1200, "points": 400}[kind]
        c.update(_survey(rng, 40, top))
        if kind in ("map", "irs") and rng.random() < 0.3:
            c["npix_y"] = max(1, int(c["npix"] * rng.uniform(0.3, 2.0)))
        if kind == "map" and rng.random() < 0.3:
            c.update(center_x=round(rng.uniform(-1, 1), 2), center_y=round(rng.uniform(-1, 1), 2))
        if kind == "map" and rng.random() < 0.2:
            c["rect"] = True
        if kind in ("map", "irs") and rng.random() < 0.5:
            c.update(leaf=rng.choice((16, 32, 64)), rows_per_item=rng.choice((64, 512)))
        if kind == "points":
            c["points"] = rng.randint(100, 100000)
        g = _geometry(c)
        if not 20 <= g["stars"] <= 200000 or g["rays"] > MAX_RAYS or g["landing"] > MAX_LANDING:
            continue
        if kind == "plain" and (g["rays"] > 4e6 or g["rays"] * g["stars"] > MAX_PAIRS):
            continue
        return c


# ---------------------------------------------------------------------------
# inputs and passes
# ---------------------------------------------------------------------------

def _stars(c, g, rng):
    """Masses (n,) and positions (n, 2), uniform in the star disk or rectangle."""
    n = g["stars"]
    if g["rect"]:
        pos = rng.uniform(-1.0, 1.0, (n, 2)) * np.array(g["rect"])
    else:
        r, phi = g["radius"] * np.sqrt(rng.random(n)), 2.0 * math.pi * rng.random(n)
        pos = np.stack([r * np.cos(phi), r * np.sin(phi)], axis=1)
    if MASSES[c["mass"]] is None:
        return np.ones(n), pos
    edges, alphas = MASSES[c["mass"]]
    weight, k0 = [], 1.0
    for k, a in enumerate(alphas):
        if k:
            k0 *= edges[k] ** (a - alphas[k - 1])
        weight.append(k0 * (edges[k + 1] ** (1 - a) - edges[k] ** (1 - a)) / (1 - a))
    seg = rng.choice(len(alphas), n, p=np.array(weight) / sum(weight))
    u, m = rng.random(n), np.empty(n)
    for k, a in enumerate(alphas):
        lo, hi = edges[k] ** (1 - a), edges[k + 1] ** (1 - a)
        m[seg == k] = (lo + u[seg == k] * (hi - lo)) ** (1.0 / (1 - a))
    return m, pos


def _args(c, g, m, pos):
    """The arguments of mm.create for a single-map case."""
    modes = {"irs": mm.MM_FMM_IRS, "plain": mm.MM_PLAIN_FP64}
    kw = {"rays_per_pixel": g["rpp"], "fmm_order": c["order"], "leaf_size": c.get("leaf", 0),
          "rows_per_item": c.get("rows_per_item", 0), "mode": modes.get(c["kind"], mm.MM_FMM_FP32),
          "img_half": g["half"], "center_y": g["centre"], "npix_y": c.get("npix_y", 0)}
    if "rays_x" in c:
        kw["ray_grid"] = g["n"]
    if g["rect"]:
        kw["star_rect"] = g["rect"]
    return (c["kappa"], c["gamma"], c["s"], m, pos, c["half_length"], c["npix"]), kw


def _points(c, g, rng):
    """Image-plane points inside the shooting region."""
    lo = np.array(g["x0"])
    return lo + rng.random((c["points"], 2)) * (np.array(g["n"]) - 1) * np.array(g["h"])


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        hs, outs = [], []
        for m in _batch_maps(case):
            g = _geometry(m)
            a, kw = _args(m, g, *_stars(m, g, rng))
            hs.append(mm.create(*a, **kw))
            outs.append(torch.empty((g["ny"], g["nx"]), dtype=torch.float32, device="cuda"))
        return {"kind": "batch", "hs": hs, "outs": outs}
    g = _geometry(case)
    m, pos = _stars(case, g, rng)
    a, kw = _args(case, g, m, pos)
    if case["kind"] == "one_shot":
        return {"kind": "one_shot", "args": a, "options": kw}
    torch.cuda.init()
    state = {"kind": case["kind"], "h": mm.create(*a, **kw)}
    if case["kind"] == "points":
        state["z"] = _points(case, g, rng)
    else:
        state["out"] = torch.empty((g["ny"], g["nx"]), dtype=torch.float32, device="cuda")
    return state


def run(state):
    if state["kind"] == "points":
        return mm.shoot_points(state["h"], state["z"])
    if state["kind"] == "batch":
        mm.run_batch(state["hs"])
        return [mm.get_map(h, out) for h, out in zip(state["hs"], state["outs"])]
    if state["kind"] == "one_shot":
        h = mm.create(*state["args"], **state["options"])
        mm.run(h)
        mu = mm.get_map(h)
        mm.destroy(h)
        return mu
    mm.run(state["h"])
    return mm.get_map(state["h"], state["out"])


def work(case):
    """Each star read and each map pixel written once; the rays that land in the map cannot be
    left out: per ray about two direct stars (11 flops each), a re-centred expansion of 0.6 times
    the order (8 flops a term), the macro model (8), and two triangles of its cell located on the
    pixel grid (20 each).  The direct sum takes 11 flops for every ray and star."""
    if case["kind"] == "batch":
        parts = [work(m) for m in _batch_maps(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    g = _geometry(case)
    ray = 22.0 + 8.0 * 0.6 * case["order"] + 8.0
    if case["kind"] == "points":
        return {"bytes": 24.0 * g["stars"] + 32.0 * case["points"], "flops": ray * case["points"]}
    out = {"bytes": 24.0 * g["stars"] + 4.0 * g["nx"] * g["ny"]}
    if case["kind"] == "plain":
        out["flops"] = g["rays"] * (11.0 * g["stars"] + 48.0)
    else:
        out["flops"] = g["landing"] * (ray + (2.0 if case["kind"] == "irs" else 40.0))
    return out


# ---------------------------------------------------------------------------
# 64-bit values
# ---------------------------------------------------------------------------

def _sources(c, g, m, pos, x, y):
    """Source positions of image points by the direct sum over every star, FP64."""
    sx, sy, sm = (torch.as_tensor(v, dtype=torch.float64, device=x.device)
                  for v in (pos[:, 0], pos[:, 1], m))
    wx, wy = torch.empty_like(x), torch.empty_like(x)
    step = max(1, int(2e7) // max(1, len(m)))
    for b in range(0, x.numel(), step):
        dx, dy = x[b:b + step, None] - sx, y[b:b + step, None] - sy
        q = sm / (dx * dx + dy * dy)
        wx[b:b + step] = (q * dx).sum(1)
        wy[b:b + step] = (q * dy).sum(1)
    k = 1.0 - c["kappa"] + g["ks"]
    return (k + c["gamma"]) * x - wx, (k - c["gamma"]) * y - wy


def _mean_clamped(a, b):
    """Mean of clamp(x, 0, 1) over x in [a, b]."""
    def prim(x):
        t = x.clamp(0.0, 1.0)
        return 0.5 * t * t + (x - 1.0).clamp(min=0.0)
    d = b - a
    flat = d < 1e-9
    return torch.where(flat, (0.5 * (a + b)).clamp(0.0, 1.0),
                       (prim(b) - prim(a)) / torch.where(flat, torch.ones_like(d), d))


def _pixel_areas(T, px, py):
    """Signed area of triangle T (k, 3, 2) inside pixel (px, py), by Green's theorem on the
    boundary clamped to the pixel."""
    tot = torch.zeros_like(px)
    for e in range(3):
        x0, y0 = T[:, e, 0] - px, T[:, e, 1] - py
        x1, y1 = T[:, (e + 1) % 3, 0] - px, T[:, (e + 1) % 3, 1] - py
        ys, ye = y0.clamp(0.0, 1.0), y1.clamp(0.0, 1.0)
        dy = y1 - y0
        slope = torch.where(dy != 0, (x1 - x0) / torch.where(dy != 0, dy, torch.ones_like(dy)),
                            torch.zeros_like(dy))
        xs, xe = x0 + (ys - y0) * slope, x0 + (ye - y0) * slope
        tot += (ye - ys) * _mean_clamped(torch.minimum(xs, xe), torch.maximum(xs, xe))
    return tot


def _polygon_map(g, u, v):
    """Sum over the cells' triangles of their area fraction per pixel; u, v: the mapped grid
    (rows, columns) in pixels."""
    nx, ny = g["nx"], g["ny"]
    acc = torch.zeros(nx * ny, dtype=torch.float64, device=u.device)
    p = torch.stack([u, v], dim=-1)
    a, b, c, d = p[:-1, :-1], p[:-1, 1:], p[1:, 1:], p[1:, :-1]
    for T in (torch.stack([a, b, c], -2), torch.stack([a, c, d], -2)):
        T = T.reshape(-1, 3, 2)
        lo, hi = T.amin(1).floor(), T.amax(1).floor()
        T, lo, hi = (t[(hi >= 0).all(1) & (lo[:, 0] < nx) & (lo[:, 1] < ny)] for t in (T, lo, hi))
        area = 0.5 * ((T[:, 1, 0] - T[:, 0, 0]) * (T[:, 2, 1] - T[:, 0, 1])
                      - (T[:, 2, 0] - T[:, 0, 0]) * (T[:, 1, 1] - T[:, 0, 1]))
        lo.clamp_(min=0.0)
        hi = torch.minimum(hi, torch.tensor([nx - 1.0, ny - 1.0], dtype=hi.dtype, device=hi.device))
        w = (hi - lo + 1).long()
        cnt = w[:, 0] * w[:, 1]
        ends = torch.cumsum(cnt, 0)
        total, at = int(ends[-1]) if len(ends) else 0, 0
        while at < total:
            stop = min(total, at + 4000000)
            k = torch.arange(at, stop, device=u.device)
            t = torch.searchsorted(ends, k, right=True)
            r = k - (ends[t] - cnt[t])
            px, py = lo[t, 0] + r % w[t, 0], lo[t, 1] + torch.div(r, w[t, 0], rounding_mode="floor")
            acc.index_add_(0, (py * nx + px).long(), _pixel_areas(T[t], px, py) / area[t])
            at = stop
    return acc


def exact(case, seed):
    if case["kind"] == "batch":
        return None
    g = _geometry(case)
    size = case.get("points", g["rays"])
    if g["rect"] or size > 3e6 or size * g["stars"] > 2e9:
        return None
    rng = np.random.default_rng(seed)
    m, pos = _stars(case, g, rng)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "points":
        z = torch.as_tensor(_points(case, g, rng), dtype=torch.float64, device=dev)
        return torch.stack(_sources(case, g, m, pos, z[:, 0], z[:, 1]), dim=1)
    x = g["x0"][0] + torch.arange(g["n"][0], dtype=torch.float64, device=dev) * g["h"][0]
    y = g["x0"][1] + torch.arange(g["n"][1], dtype=torch.float64, device=dev) * g["h"][1]
    yy, xx = torch.meshgrid(y, x, indexing="ij")
    wx, wy = _sources(case, g, m, pos, xx.reshape(-1), yy.reshape(-1))
    u = ((wx - (g["centre"][0] - g["side"][0])) / g["delta"]).reshape(yy.shape)
    v = ((wy - (g["centre"][1] - g["side"][1])) / g["delta"]).reshape(yy.shape)
    cell = g["h"][0] * g["h"][1] / g["delta"] ** 2
    if case["kind"] == "irs":
        ok = (u >= 0) & (u < g["nx"]) & (v >= 0) & (v < g["ny"])
        idx = v[ok].floor().long() * g["nx"] + u[ok].floor().long()
        mu = torch.bincount(idx, minlength=g["nx"] * g["ny"]).to(torch.float64) * cell
    else:
        mu = _polygon_map(g, u, v) * (0.5 * cell)
    return mu.reshape(g["ny"], g["nx"])
