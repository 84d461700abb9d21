"""Timed cases of the shallow-water library: what a user's program asks of it, through its
public entry points.

Every case is one whole piece of work: a run is the initial state handed over, the steps,
and the read-outs that such a program takes; a gradient is the forward run and its backward;
the depth filter is one call. Grids, bathymetry and record buffers are made beforehand, as a
program that runs several sources on one grid keeps them. The shapes are those of the
repository's configurations (`workloads/`: the beach, the geographic coast, the shelf with
islands, the ensemble basin, the inversion, the run-up line), drawn from the seed.

`exact` restates the scheme in plain torch FP64, whole fields at a time, and differentiates it
with torch.autograd.
"""
import math

import numpy as np
import torch

import paper_1410_0753_gb300 as pk
from paper_1410_0753_gb300.autograd import gauge_run

G = 9.81
R_EARTH = 6371000.0
MANNING_N2 = 0.025 ** 2
H_MIN = 0.01


def _case(name=None, **kw):
    c = dict(kind="forward", bathy="beach", nx=200, ny=200, steps=200, batch=1, friction=True, transverse=1,
             alternate=0, open_edges=0, itopo=1, maxout=0, gout=1, checkpoint=0, persistent=False, nests=0)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the run-up of a solitary wave on a 1D line (the benchmark problem of the method):
        # the smallest call, a chain of launches over a few hundred nodes
        _case("runup line", kind="line", bathy="line", nx=613, ny=1, steps=300, friction=False, maxout=1),
        # a small 2D run with every output due, as in the quick start: latency of one step
        _case("beach 200", bathy="beach", nx=200, ny=200, steps=200, maxout=1),
        # one scenario on the ensemble's grid: a mid-size grid that alone does not fill the GPU
        _case("basin 512", bathy="basin", nx=512, ny=512, steps=120, maxout=20),
        # the same small grid in one persistent launch
        _case("basin 300x257 persistent", bathy="basin", nx=300, ny=257, steps=200, maxout=20, persistent=True),
        # a child grid of a nesting chain, driven by boundary series on three edges, geographic
        _case("nested child 331x287", kind="child", bathy="coast", nx=331, ny=287, steps=120, maxout=1),
        # an odd-sized open domain with radiating edges and the alternating sweep order
        _case("open 1201x901", bathy="basin", nx=1201, ny=901, steps=40, open_edges=13, alternate=1, gout=4),
        # the regional model: geographic metric, max-wave, gauges and enclosed grids every step
        _case("coast 2048", bathy="coast", nx=2048, ny=2048, steps=24, maxout=1, nests=2),
        # the large domain, no outputs during the run
        _case("shelf 8192", bathy="shelf", nx=8192, ny=8192, steps=12),
        # scenarios of uneven durations on one bathymetry in one launch
        _case("ensemble 48x512", kind="ensemble", bathy="basin", nx=512, ny=512, batch=48, steps=120, persistent=True),
        # source inversion: forward and gradient through autograd, every state kept
        _case("inversion 1024", kind="gradient", bathy="basin", nx=1024, ny=1024, steps=48),
        # a gradient with checkpoints (states recomputed), odd sizes, geographic
        _case("gradient 613x447", kind="gradient", bathy="coast", nx=613, ny=447, steps=120, checkpoint=20),
        # the depth-jump filter into the caller's memory, the step before every run
        _case("depth filter 1000", kind="filter", bathy="rough", nx=1000, ny=1000, steps=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges; every one costs less than the largest listed."""
    kind = rng.choice(["forward", "forward", "forward", "line", "child", "ensemble", "gradient", "filter"])
    if kind == "line":
        return _case(kind="line", bathy="line", nx=_log(rng, 300, 4000), ny=1, steps=_log(rng, 100, 600),
                     friction=False, maxout=rng.choice([1, 10]))
    if kind == "filter":
        return _case(kind="filter", bathy="rough", nx=_log(rng, 60, 1024), ny=_log(rng, 60, 1024), steps=1)
    nx, ny = _log(rng, 90, 900), _log(rng, 90, 900)
    opts = dict(friction=rng.random() < 0.8, transverse=int(rng.random() < 0.9))
    if kind == "child":
        return _case(kind="child", bathy="coast", nx=nx, ny=ny, steps=_log(rng, 30, 160),
                     maxout=rng.choice([1, 10]), persistent=rng.random() < 0.5, **opts)
    if kind == "ensemble":
        batch = _log(rng, 2, 48)
        nx, ny = _log(rng, 90, 512), _log(rng, 90, 512)
        return _case(kind="ensemble", bathy=rng.choice(["basin", "beach"]), nx=nx, ny=ny, batch=batch,
                     steps=_log(rng, 30, 120), persistent=rng.random() < 0.8, **opts)
    if kind == "gradient":
        return _case(kind="gradient", bathy=rng.choice(["basin", "coast", "beach"]), nx=nx, ny=ny,
                     steps=_log(rng, 20, 100), checkpoint=rng.choice([0, 0, 10, 25]), **opts)
    nx, ny = _log(rng, 90, 6000), _log(rng, 90, 6000)
    steps = max(8, min(200, int(6.0e8 / (nx * ny))))
    bathy = rng.choice(["beach", "basin", "coast", "shelf"])
    return _case(bathy=bathy, nx=nx, ny=ny, steps=steps, maxout=rng.choice([0, 1, 10]),
                 alternate=int(rng.random() < 0.15), open_edges=rng.choice([0, 0, 0, 5, 15]),
                 persistent=rng.random() < 0.3, nests=rng.choice([0, 0, 1]) if bathy == "coast" else 0, **opts)


# ------------------------------------------------------------------ inputs

def _f32(a):
    return a.to(torch.float32).to(torch.float64)


def _waves(rng, X, Y, nx, ny, n=10):
    """A smooth random field of about unit size: plane waves of the domain's length scales."""
    out = torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    for _ in range(n):
        k = 2 * math.pi * rng.uniform(1.0, 12.0)
        th = rng.uniform(0, 2 * math.pi)
        out += (math.sqrt(2.0 / n)) * torch.cos(k * math.cos(th) * X + k * math.sin(th) * Y + rng.uniform(0, 2 * math.pi))
    return out


def _inputs(case, seed):
    """Nodes, depth, initial free surfaces, gauges, dt, and what the kind needs besides, as
    FP32-representable FP64 tensors on the GPU; the same for prepare and exact."""
    rng = np.random.default_rng([seed, 1410, case["nx"], case["ny"]])
    nx, ny = case["nx"], case["ny"]
    f64 = dict(dtype=torch.float64, device="cuda")
    s = dict(rng=rng, coords=1)
    if case["kind"] == "line":
        # deep water, a plane beach 1:19.85 up through the still shoreline, spacing refined
        slope, H = 19.85, rng.uniform(0.012, 0.03)
        gam = math.sqrt(0.75 * H)
        toe = -slope
        x1 = toe - 1.2 * math.acosh(math.sqrt(20.0)) / gam
        w = np.concatenate([np.linspace(1.0, 0.25, nx // 3), np.full(nx - 1 - nx // 3, 0.25)])
        x = np.concatenate([[0.0], np.cumsum(w)])
        x = 3.0 - 70.0 * (1.0 - x / x[-1])
        x = torch.as_tensor(x, **f64)
        d = torch.where(x <= toe, torch.ones_like(x), -x / slope)
        eta = torch.where(d > 0, H / torch.cosh(gam * (x - x1)) ** 2, torch.zeros_like(x))
        s.update(x=_f32(x), y=torch.zeros(1, **f64), d=_f32(d[None]), eta0=_f32(eta[None]),
                 u0=_f32((eta * math.sqrt(G))[None]), h_min=0.003, gauges=[])
        ds = float((s["x"][1:] - s["x"][:-1]).min())
        s["dt"] = 0.7 * ds / math.sqrt(G * 1.05)
        return s
    X = (torch.arange(nx, **f64) / max(nx - 1, 1))[None, :]
    Y = (torch.arange(ny, **f64) / max(ny - 1, 1))[:, None]
    b = case["bathy"]
    if case["kind"] == "filter":
        # steep synthetic relief: a rough sea floor with land, many violations of the limit
        d = 300.0 * torch.exp(1.5 * _waves(rng, X, Y, nx, ny)) - 150.0
        gen = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7fffffff)
        d = d * torch.exp(0.5 * torch.randn(ny, nx, generator=gen, **f64))
        s.update(d=d.contiguous())
        return s
    noise = _waves(rng, X, Y, nx, ny)
    if b == "beach":            # 50 m offshore, then a plane beach to +10 m, 100 m spacing
        dx = 100.0
        d = torch.where(X <= 0.5, torch.full_like(X, 50.0), 50.0 - 120.0 * (X - 0.5)) * torch.ones_like(Y)
        d = d * (1.0 + 0.03 * noise)
    elif b == "basin":          # 3000 m, slope to the shore at 0.93, land to +20 m, 200 m spacing
        dx = 200.0
        d = torch.where(X <= 0.5, torch.full_like(X, 3000.0), 3000.0 * (0.93 - X) / 0.43)
        d = torch.where(X > 0.93, -20.0 * (X - 0.93) / 0.07, d) * torch.ones_like(Y)
        d = d * (1.0 + 0.02 * noise)
    elif b == "coast":          # geographic: land in the west, shelf, slope, 4000 m plain
        s["coords"] = 0
        dx = None
        shore = 0.12 + 0.03 * torch.sin(2 * math.pi * Y * rng.uniform(1.0, 2.5) + rng.uniform(0, 6)) + 0.01 * noise
        r = X - shore
        d = torch.where(r < 0, torch.clamp(400.0 * r, min=-50.0), torch.clamp(6000.0 * r, max=150.0))
        d = d + torch.clamp((r - 0.12) / 0.15, 0.0, 1.0) * 3850.0
        d = d * (1.0 + 0.05 * noise)
    else:                       # a 200 m shelf with conical islands, 50 m spacing
        dx = 50.0
        d = 200.0 * (1.0 + 0.04 * noise)
        for _ in range(10):
            cx, cy = rng.uniform(0.3, 0.95), rng.uniform(0.3, 0.95)
            rb, top = rng.uniform(0.01, 0.05), rng.uniform(20.0, 80.0)
            r = torch.sqrt((X - cx) ** 2 + ((Y - cy) * ny / nx) ** 2) / rb
            d = torch.minimum(d, -top + (200.0 + top) * r)
    if s["coords"] == 1:
        s["x"], s["y"] = _f32(torch.arange(nx, **f64) * dx), _f32(torch.arange(ny, **f64) * dx)
        ds = dx
    else:
        s["x"], s["y"] = _f32(140.0 + torch.arange(nx, **f64) / 60.0), _f32(20.0 + torch.arange(ny, **f64) / 60.0)
        ds = R_EARTH * math.cos(math.radians(float(s["y"][-1]))) * math.radians(1.0 / 60.0) * 0.999
    s["d"] = _f32(d)
    s["h_min"] = H_MIN
    dmax = float(s["d"].max())
    s["dt"] = rng.uniform(0.6, 0.8) * ds / math.sqrt(G * dmax)
    # sources: Gaussian humps in deep water
    nb = case["batch"]
    eta = torch.zeros(nb, ny, nx, **f64)
    lo, hi = {"beach": (0.25, 0.6), "basin": (0.15, 0.55), "coast": (0.4, 0.8), "shelf": (0.1, 0.3)}[b]
    for k in range(nb):
        for _ in range(2):
            cx, cy, sg = rng.uniform(lo, hi), rng.uniform(0.2, 0.8), rng.uniform(0.04, 0.09)
            a = rng.uniform(0.3, 1.0)
            eta[k] += a * torch.exp(-((X - cx) ** 2 + (Y - cy) ** 2) / (2 * sg * sg))
    eta = torch.where(s["d"] > 0, eta, torch.zeros_like(eta))
    s["eta0"] = _f32(eta if case["kind"] == "ensemble" else eta[0])
    gx = np.clip((np.array([0.3, 0.45, 0.6, 0.75]) * nx).astype(int), 0, nx - 1)
    gy = np.clip((np.array([0.15, 0.4, 0.6, 0.85]) * ny).astype(int), 0, ny - 1)
    s["gauges"] = [(int(i), int(j)) for i in gx for j in gy]
    if case["nests"]:
        s["nests"] = [pk.cliffs_nest(float(s["x"][nx // 5]), float(s["y"][ny * (1 + 2 * k) // 6]),
                                     1.0 / 180.0, 1.0 / 180.0, min(301, 2 * nx // 3), min(301, 2 * ny // 7))
                      for k in range(case["nests"])]
    if case["kind"] == "child":
        # series on the east, south and north edges: a plane wave train rising from rest and
        # running toward the shore
        nt, dtr = case["steps"] // 4 + 3, 4.0 * s["dt"]
        t = torch.arange(nt, **f64) * dtr
        om, amp = 2 * math.pi / (40.0 * s["dt"]), rng.uniform(0.2, 0.6)
        ks = rng.uniform(2.0, 4.0)
        s["series"] = {}
        for e, (px, py, dd) in {1: (0.0 * Y[:, 0] + 1.0, Y[:, 0], s["d"][:, -1]), 2: (X[0], 0.0 * X[0], s["d"][0]),
                                3: (X[0], 0.0 * X[0] + 1.0, s["d"][-1])}.items():
            ramp = torch.clamp(t / (20.0 * s["dt"]), max=1.0)[:, None]
            el = amp * ramp * torch.sin(om * t[:, None] + ks * (px - 1.0 + 0.3 * py)[None])
            el = torch.where(dd[None] > 20.0, el, torch.zeros_like(el))
            uu = -el * torch.sqrt(G / torch.clamp(dd, min=20.0))[None]
            s["series"][e] = (t, torch.stack([uu, 0.3 * uu, el], dim=1).contiguous())
        s["eta0"] = torch.zeros_like(s["eta0"])
    if case["kind"] == "ensemble":
        n = case["steps"]
        s["durations"] = rng.integers(max(1, n // 6), n + 1, nb).astype(np.int64)
        s["durations"][int(rng.integers(nb))] = n
    if case["kind"] == "gradient":
        nrec = case["steps"] + 1
        ph = rng.uniform(0, 6, len(s["gauges"]))
        s["seed"] = torch.as_tensor(0.1 * np.sin(0.2 * np.arange(nrec)[:, None] + ph[None, :]), **f64).to(torch.float32)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    st = {"case": case}
    if case["kind"] == "filter":
        st["depth"] = s["d"]
        st["out"] = torch.empty_like(s["d"])
        return st
    n, nb = case["steps"], case["batch"]
    g = pk.CliffsGrid(case["nx"], case["ny"], s["dt"], batch=nb, coords=s["coords"], h_min=s["h_min"],
                      manning_n2=MANNING_N2 if case["friction"] else 0.0, itopo=case["itopo"],
                      transverse=case["transverse"], alternate=case["alternate"], maxout=case["maxout"] or n + 1,
                      gout=case["gout"], gauges=s["gauges"], nests=s.get("nests", ()), open_edges=case["open_edges"])
    g.set_bathy(s["x"].cpu().numpy(), s["y"].cpu().numpy(), s["d"], case["kind"] != "line")
    st["grid"] = g
    st["eta0"] = s["eta0"].to(torch.float32).contiguous()
    st["u0"] = s["u0"].to(torch.float32).contiguous() if "u0" in s else None
    shape = (case["ny"], case["nx"])
    if case["maxout"]:
        st["maxwave"] = [torch.empty(shape, device="cuda"), torch.empty(shape, device="cuda")]
    for e, (t, v) in s.get("series", {}).items():
        g.set_boundary_input(e, t.cpu().numpy(), v)
    if "series" in s:
        g.set_boundary_clock()
    if case["kind"] == "ensemble":
        st["durations"] = s["durations"]
        st["states"] = torch.empty((nb, 3) + shape, device="cuda")
        st["records"] = torch.zeros((nb, n + 1, len(s["gauges"]), 3), device="cuda")
        g.set_initial(st["eta0"])
        g.set_durations(s["durations"])
    if case["kind"] == "gradient":
        st["seed"] = s["seed"]
    return st


def run(st):
    case = st["case"]
    if case["kind"] == "filter":
        passes = pk.cliffs_depth_filter_noalloc(st["depth"], st["out"], case["nx"], case["ny"])
        return {"depth": st["out"], "passes": passes}
    g = st["grid"]
    if case["kind"] == "gradient":
        eta0 = st["eta0"].detach().requires_grad_(True)
        rec = gauge_run(eta0, g, case["steps"], case["checkpoint"] or None)
        rec.backward(st["seed"])
        return {"records": rec.detach(), "gradient": eta0.grad}
    g.set_initial(st["eta0"], st["u0"])
    g.step(case["steps"], persistent=case["persistent"])
    if case["kind"] == "ensemble":
        for b in range(case["batch"]):
            pk.cliffs_read_state(g.h, b, st["states"][b, 0], st["states"][b, 1], st["states"][b, 2])
            pk.cliffs_read_gauges(g.h, b, st["records"][b])
        return {"state": st["states"], "records": st["records"]}
    out = {"state": list(g.state_views())}
    if g.n_gauges:
        out["gauges"] = g.gauges()
    if case["maxout"]:
        pk.cliffs_read_maxwave(g.h, 0, st["maxwave"][0], st["maxwave"][1])
        # nodes that were never wet hold the type's lowest value: cut off for a map
        out["maxwave"] = [st["maxwave"][0].clamp(min=-1.0), st["maxwave"][1]]
    if case["nests"]:
        # the series an enclosed grid is driven with, stored in single precision
        out["boundary"] = [g.boundary(0, e).astype(np.float32) for e in range(4)]
    return out


def work(case):
    cells = case["nx"] * case["ny"] * case["batch"]
    if case["kind"] == "filter":
        return {"bytes": 16.0 * cells, "flops": 8.0 * cells}
    n = case["steps"] * (0.58 if case["kind"] == "ensemble" else 1.0)
    sweeps = 1 if case["kind"] == "line" else 2
    flops = (75.0 if case["friction"] else 60.0) * sweeps * cells * n      # one sweep of one node
    if case["kind"] == "gradient":
        flops *= 4.0                                            # the run, and the transpose of each step
        return {"bytes": cells * 12.0, "flops": flops}          # eta0 and d in, the gradient out
    byts = cells * (4.0 + 12.0 + (8.0 if case["maxout"] else 0.0)) + case["nx"] * case["ny"] * 4.0
    return {"bytes": byts, "flops": flops}


# ------------------------------------------------------------------ the scheme in FP64

def _filter(d, alpha=2.0, dmin=0.1):
    """The depth-jump filter: rows then columns, Jacobi, until nothing changes."""
    a2 = alpha * alpha
    d = torch.where((d > 0) & (d < dmin), torch.full_like(d, dmin), d)
    for k in range(1, 101):
        before = d
        for dim in (1, 0):
            n = d.shape[dim]
            if n < 3:
                continue
            i = torch.arange(n, device=d.device)
            i = i[None, :] if dim == 1 else i[:, None]
            l, r = torch.roll(d, 1, dim), torch.roll(d, -1, dim)
            wl, wr = (i > 0) & (l > 0), (i < n - 1) & (r > 0)
            viol = (d > 0) & ((wl & (l > a2 * d)) | (wr & (r > a2 * d)))
            mean = (torch.sqrt(l.clamp(min=0)) + torch.sqrt(r.clamp(min=0))) ** 2 / 4.0
            d = torch.where(viol, torch.where(wl & wr, mean, torch.where(wl, l, r) / a2), d)
        if torch.equal(before, d):
            return d, k
    return d, -1


def _flux(a, b):
    (ea, wa, ta, da, ca), (eb, wb, tb, db, cb) = a, b
    dc = G * ((eb - ea) + (db - da)) / (cb + ca)
    sw, sc, dw = wb + wa, cb + ca, wb - wa
    z = G * (eb - ea)
    return 0.5 * dw * (sw + sc) + z + sw * dc, 0.5 * dw * (sw - sc) + z - sw * dc, 0.5 * sw * (tb - ta)


def _sweep(P, e, w, t, d, il, ir, k2, sdt, lo, hi):
    """One sweep along the last axis: marks, flooding, walls, eq. (solver2), cushion."""
    dt, hm = P["dt"], P["h_min"]
    n = e.shape[-1]
    i = torch.arange(n, device=e.device)
    first, last = i == 0, i == n - 1
    L = lambda x: torch.roll(x, 1, -1)      # noqa: E731
    R = lambda x: torch.roll(x, -1, -1)     # noqa: E731
    zero, one = torch.zeros_like(e), torch.ones_like(e)
    floor = d >= P["dwall"]
    o = floor & (e + d >= hm)
    w, t = torch.where(o, w, zero), torch.where(o, t, zero)
    oL, oR = L(o) & ~first, R(o) & ~last
    okL, okR = ~o & floor & oL & (L(e) + d > hm), ~o & floor & oR & (R(e) + d > hm)
    useR = okR & (~okL | (R(e) > L(e)))
    fl = okL | okR
    e, w, t = (torch.where(fl, hm - d, e), torch.where(fl, torch.where(useR, R(w), L(w)), w),
               torch.where(fl, torch.where(useR, R(t), L(t)), t))
    wet = o | fl
    c = torch.sqrt(torch.where(wet, G * (e + d), one))
    C = (e, w, t, d, c)
    mirror = (e, -w, t, d, c)
    wl, wr = L(wet) & ~first, R(wet) & ~last
    left = tuple(torch.where(wl, L(x), m) for x, m in zip(C, mirror))
    right = tuple(torch.where(wr, R(x), m) for x, m in zip(C, mirror))

    def ghost(s):
        c0 = torch.sqrt(torch.where(d > 0, G * d, one)) * (d > 0)
        delta = c - c0
        cg = torch.clamp(c + s * 0.25 * w - 0.5 * delta, min=0.0)
        return cg * cg / G - d, 0.5 * w + s * delta, t, d, cg

    if lo:
        left = tuple(torch.where(first & wet, g, x) for g, x in zip(ghost(-1.0), left))
    if hi:
        right = tuple(torch.where(last & wet, g, x) for g, x in zip(ghost(1.0), right))
    pl, ql, tl = (f * il for f in _flux(left, C))
    pr, qr, tr = (f * ir for f in _flux(C, right))
    dp = -0.5 * dt * (pl + pr) + (w + c) * k2 * (pr - pl)
    dq = -0.5 * dt * (ql + qr) + (w - c) * k2 * (qr - ql)
    if P["n2"] > 0:
        h = torch.where(wet, e + d, one)
        s2 = w * w + t * t
        sp = torch.where(s2 > 0, torch.sqrt(torch.where(s2 > 0, s2, one)), zero)
        adt = w * torch.clamp(dt * G * P["n2"] * sp * h ** (-4.0 / 3.0), max=1.0)
        dp, dq = dp - adt, dq - adt
    if sdt is not None:
        dp, dq = dp + sdt * c * w, dq - sdt * c * w
    dc = 0.25 * (dp - dq)
    e2 = torch.where(wet, e + dc * (2 * c + dc) / G, e)
    w2 = torch.where(wet, w + 0.5 * (dp + dq), w)
    t2 = t
    if P["transverse"]:
        t2 = torch.where(wet, t - 0.5 * dt * (tl + tr) + w * k2 * (tr - tl), t)
    hs, ws = torch.where(useR, R(e2 + d), L(e2 + d)), torch.where(useR, R(w2), L(w2))
    e3 = torch.where(fl & (e2 + d > 0.5 * hs), 0.5 * hs - d, e2)
    w3 = torch.where(fl & (w2.abs() > ws.abs()), ws, w2)
    return e3, w3, t2


def _metric(P, s, case):
    dt = P["dt"]

    def axis(c, f):
        if len(c) == 1:
            return None
        h = f * (c[1:] - c[:-1])
        l, r = torch.cat([h[:1], h]), torch.cat([h, h[-1:]])
        return 1.0 / l, 1.0 / r, dt * dt / (l + r)

    if s["coords"] == 1:
        return axis(s["x"], 1.0), axis(s["y"], 1.0), None
    rad = math.pi / 180.0
    x = axis(s["x"], rad)
    f = (1.0 / (R_EARTH * torch.cos(s["y"] * rad)))[:, None]
    return tuple(v[None] * f for v in x), axis(s["y"], R_EARTH * rad), dt * torch.tan(s["y"] * rad) / R_EARTH


def _step(P, M, e, u, v, d, yfirst):
    mx, my, sdt = M
    oe = P["open"]

    def xs(e, u, v):
        return _sweep(P, e, u, v, d, *mx, None, oe & 1, oe & 2) if mx is not None else (e, u, v)

    def ys(e, u, v):
        if my is None:
            return e, u, v
        T = lambda q: q.transpose(-1, -2)   # noqa: E731
        a, b, c = _sweep(P, T(e), T(v), T(u), T(d), *my, sdt, oe & 4, oe & 8)
        return T(a), T(c), T(b)

    return xs(*ys(e, u, v)) if yfirst else ys(*xs(e, u, v))


def _impose(s, t, e, u, v):
    e, u, v = e.clone(), u.clone(), v.clone()
    for k, (T, V) in s["series"].items():
        Th = T.cpu().numpy()
        i = int(np.clip(np.searchsorted(Th, t, side="right") - 1, 0, len(Th) - 1))
        w = 0.0 if i == len(Th) - 1 else (t - Th[i]) / (Th[i + 1] - Th[i])
        val = (1.0 - w) * V[i] + (w * V[i + 1] if w > 0 else 0.0)
        at = (slice(None), 0) if k == 0 else (slice(None), -1) if k == 1 else (0,) if k == 2 else (-1,)
        u[at], v[at], e[at] = val[0], val[1], val[2]
    return e, u, v


def _wet(P, e, d):
    return (d >= P["dwall"]) & (e + d >= P["h_min"])


def exact(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "filter":
        d, k = _filter(s["d"])
        return {"depth": d, "passes": None}
    P = dict(dt=s["dt"], h_min=s["h_min"], n2=MANNING_N2 if case["friction"] else 0.0, open=case["open_edges"],
             transverse=case["transverse"], dwall=-math.inf if case["itopo"] else 0.0)
    d = s["d"] if case["kind"] == "line" else _filter(s["d"])[0]
    M = _metric(P, s, case)
    n = case["steps"]
    gx = torch.tensor([g[0] for g in s["gauges"]], device="cuda", dtype=torch.long)
    gy = torch.tensor([g[1] for g in s["gauges"]], device="cuda", dtype=torch.long)
    e = s["eta0"]
    u = s.get("u0", torch.zeros_like(e))
    v = torch.zeros_like(e)

    def pick(e, u, v):
        return torch.stack([q[..., gy, gx] for q in (e, u, v)], dim=-1)

    if case["kind"] == "gradient":
        states, recs = [(e, u, v)], [e[gy, gx]]
        for j in range(n):
            states.append(_step(P, M, *states[-1], d, case["alternate"] and j & 1))
            recs.append(states[-1][0][gy, gx])
        seed_ = s["seed"].double()
        lam = [torch.zeros_like(e) for _ in range(3)]
        lam[0].index_put_((gy, gx), seed_[n], accumulate=True)
        for j in range(n - 1, -1, -1):
            x = [q.detach().requires_grad_(True) for q in states[j]]
            y = _step(P, M, *x, d, case["alternate"] and j & 1)
            lam = list(torch.autograd.grad(y, x, grad_outputs=lam))
            lam[0] = lam[0].index_put((gy, gx), seed_[j], accumulate=True)
        return {"records": torch.stack(recs), "gradient": lam[0]}
    if case["kind"] == "ensemble":
        dur = torch.as_tensor(s["durations"], device="cuda")
        rec = torch.zeros((case["batch"], n + 1, len(gx), 3), dtype=torch.float64, device="cuda")
        rec[:, 0] = pick(e, u, v)
        for j in range(n):
            on = (dur > j)[:, None, None]
            new = _step(P, M, e, u, v, d, case["alternate"] and j & 1)
            e, u, v = (torch.where(on, a, b) for a, b in zip(new, (e, u, v)))
            rec[:, j + 1] = torch.where(on[..., None][:, 0], pick(e, u, v), rec[:, j + 1])
        return {"state": torch.stack([e, u, v], dim=1), "records": rec}
    every = case["maxout"] or n + 1
    low = torch.full_like(e, -1.0)
    wet = _wet(P, e, d)
    em, sm = torch.where(wet, e, low), torch.where(wet, torch.sqrt(u * u + v * v), torch.zeros_like(e))
    recs = [pick(e, u, v)]
    for j in range(n):
        if "series" in s:
            e, u, v = _impose(s, j * s["dt"], e, u, v)
        e, u, v = _step(P, M, e, u, v, d, case["alternate"] and j & 1)
        if (j + 1) % every == 0 or (j + 1 == n and case["maxout"]):
            wet = _wet(P, e, d)
            em = torch.where(wet, torch.maximum(em, e), em)
            sm = torch.where(wet, torch.maximum(sm, torch.sqrt(u * u + v * v)), sm)
        if (j + 1) % case["gout"] == 0:
            recs.append(pick(e, u, v))
    out = {"state": [e, u, v]}
    if len(gx):
        out["gauges"] = torch.stack(recs)
    if case["maxout"]:
        out["maxwave"] = [em, sm]
    if case["nests"]:
        out["boundary"] = [None] * 4
    return out
