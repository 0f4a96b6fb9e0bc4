"""What this library's users run, as measurable cases.

Every case is one whole call (or a burst of calls) through the public entry
points of ``paper_1204_6630_gb300.tpcf`` on synthetic catalogs of the shapes the
package's own generators describe (clustered data, uniform randoms), drawn here
on the GPU so that inputs of many sizes and seeds are quick to make.

Operations (``op``):
  correlate  host arrays in, (DD, DR, RR, w) out: preparation, counting, estimator
  count      DD, DR and RR of two prepared catalogs, one call (``part``: all, auto, cross)
  graph      a captured auto count, replayed
  patches    per-patch DD, DR, RR of two segmented catalogs (jackknife patches)
  jackknife  leave-one-out histograms, w and its covariance
  box        3-D distances: DD, DR and RR of two prepared 3-D catalogs
  serve      a burst of jobs through the job server (submit all, wait for all)
"""
import math

import numpy as np
import torch

from paper_1204_6630_gb300 import tpcf

DEG = math.pi / 180.0


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest job of a pair-count service: 1,000 galaxies against 2,000 randoms in a
        # 15 degree cap, host arrays in and w(theta) out; launches, copies and host work count
        {"name": "correlate_1k", "op": "correlate", "nd": 1000, "nr": 2000, "sky": "cap", "radius": 15.0,
         "bins": "lin", "lo": 0.0, "hi": 2.0, "nb": 20},
        # a survey tile of ordinary size from host arrays, sizes no multiple of anything:
        # preparation (upload, sort, copies) beside the count
        {"name": "correlate_100k", "op": "correlate", "nd": 100003, "nr": 200006, "sky": "cap", "radius": 20.0,
         "bins": "lin", "lo": 0.0, "hi": 2.0, "nb": 50},
        # a small problem on resident catalogs (the 8192-point octant workload): one count in a loop
        {"name": "octant_8k", "op": "count", "part": "all", "nd": 8192, "nr": 8192, "sky": "octant", "clusters": 128,
         "sigma": 0.5, "bins": "lin", "lo": 0.0, "hi": 10.0, "nb": 40, "mode": "screen"},
        # the headline workload: a million galaxies and a million randoms on an octant, 64 log bins
        {"name": "octant_1m", "op": "count", "part": "all", "nd": 1000000, "nr": 1000000, "sky": "octant",
         "clusters": 1024, "sigma": 0.2, "bins": "log", "lo": 0.01, "hi": 10.0, "nb": 64, "mode": "screen"},
        # the cross count of a full-sky catalog against its randoms at small angles: nearly every
        # pair is out of range (the large full-sphere workload's shape at a size that fits here)
        {"name": "sphere_cross", "op": "count", "part": "cross", "nd": 700001, "nr": 1400003, "sky": "sphere",
         "clusters": 4096, "sigma": 0.1, "bins": "log", "lo": 0.005, "hi": 2.0, "nb": 80, "mode": "screen"},
        # the same sky with spatial pruning switched on (TPCF_F_PRUNE), where users put their largest catalogs
        {"name": "sphere_prune", "op": "count", "part": "all", "nd": 1500000, "nr": 3000000, "sky": "sphere",
         "clusters": 4096, "sigma": 0.1, "bins": "log", "lo": 0.005, "hi": 2.0, "nb": 80, "mode": "prune"},
        # a captured auto count replayed (a loop over one catalog, launch-bound)
        {"name": "graph_20k", "op": "graph", "nd": 20011, "sky": "octant", "clusters": 128, "sigma": 0.5,
         "bins": "log", "lo": 0.01, "hi": 10.0, "nb": 64},
        # the all-binary64 comparator, for users who want every pair in binary64
        {"name": "plain_30k", "op": "count", "part": "all", "nd": 30011, "nr": 30011, "sky": "octant",
         "clusters": 128, "sigma": 0.5, "bins": "lin", "lo": 0.0, "hi": 10.0, "nb": 40, "mode": "plain"},
        # jackknife patches: 512 patches of uneven occupancy, nearly every pair in range
        {"name": "patches_512", "op": "patches", "nd": 2000000, "patches": 512, "bins": "lin", "lo": 0.0, "hi": 5.0,
         "nb": 40},
        # the delete-one jackknife of a catalog in 64 patches
        {"name": "jackknife_64", "op": "jackknife", "nd": 200000, "patches": 64, "bins": "lin", "lo": 0.0, "hi": 5.0,
         "nb": 40},
        # the 3-D variant: a clustered box against its randoms, 30 log distance bins
        {"name": "box_300k", "op": "box", "nd": 300000, "nr": 300000, "side": 1000.0, "lo": 0.5, "hi": 50.0, "nb": 30},
        # a burst of mixed jobs through the job server, the way a service sees them
        {"name": "serve_16", "op": "serve", "jobs": 16, "nmin": 1000, "nmax": 150000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _angles(rng):
    """Bins of the angular range that the named workloads span."""
    if rng.random() < 0.5:
        return {"bins": "lin", "lo": 0.0, "hi": round(rng.uniform(1.0, 10.0), 3), "nb": rng.randint(20, 80)}
    hi = round(rng.uniform(1.0, 10.0), 3)
    return {"bins": "log", "lo": round(hi / rng.choice([100.0, 400.0, 1000.0]), 5), "hi": hi, "nb": rng.randint(20, 80)}


def draw(rng):
    op = rng.choice(["correlate", "correlate", "count", "count", "count", "count", "graph", "patches", "jackknife",
                     "box", "serve"])
    if op == "correlate":
        nd = _log(rng, 1000, 300000)
        return {"op": op, "nd": nd, "nr": 2 * nd, "sky": "cap", "radius": round(rng.uniform(5.0, 30.0), 2),
                "bins": "lin", "lo": 0.0, "hi": 2.0, "nb": rng.randint(20, 80)}
    if op == "count":
        sky = rng.choice(["octant", "sphere"])
        mode = rng.choice(["screen", "screen", "screen", "prune", "prune", "plain", "check"])
        nd = _log(rng, 2000, {"plain": 40000, "prune": 1200000}.get(mode, 700000))
        return {"op": op, "part": rng.choice(["all", "auto", "cross"]), "nd": nd, "nr": int(nd * rng.choice([1, 1.5, 2])),
                "sky": sky, "clusters": 1024, "sigma": rng.choice([0.1, 0.2, 0.5]), "mode": mode, **_angles(rng)}
    if op == "graph":
        return {"op": op, "nd": _log(rng, 2000, 300000), "sky": rng.choice(["octant", "sphere"]), "clusters": 256,
                "sigma": 0.3, **_angles(rng)}
    if op == "patches":
        p = rng.choice([32, 64, 128, 512])
        return {"op": op, "nd": p * _log(rng, 500, 4000), "patches": p, "bins": "lin", "lo": 0.0,
                "hi": round(rng.uniform(2.0, 8.0), 2), "nb": rng.randint(20, 60)}
    if op == "jackknife":
        p = rng.choice([16, 33, 64, 100])
        return {"op": op, "nd": p * _log(rng, 300, 2500), "patches": p, "bins": "lin", "lo": 0.0,
                "hi": round(rng.uniform(2.0, 8.0), 2), "nb": rng.randint(20, 60)}
    if op == "box":
        nd = _log(rng, 5000, 400000)
        return {"op": op, "nd": nd, "nr": int(nd * rng.choice([1, 2])), "side": 1000.0, "lo": 0.5,
                "hi": round(rng.uniform(20.0, 80.0), 2), "nb": rng.randint(20, 40)}
    return {"op": op, "jobs": rng.randint(4, 20), "nmin": 1000, "nmax": rng.choice([20000, 60000, 150000])}


# ------------------------------------------------------------------ inputs
def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1000003 + k) % (1 << 62))


def _rand(g, *n):
    return torch.rand(*n, generator=g, device="cuda", dtype=torch.float64)


def _tangent(c):
    """Unit vectors along increasing RA and Dec at the unit vectors c."""
    rho = torch.sqrt(c[:, 0] ** 2 + c[:, 1] ** 2).clamp_min(1e-300)
    ca, sa = c[:, 0] / rho, c[:, 1] / rho
    e_a = torch.stack([-sa, ca, torch.zeros_like(ca)], 1)
    e_d = torch.stack([-c[:, 2] * ca, -c[:, 2] * sa, rho], 1)
    return e_a, e_d


def _uniform(n, sky, radius, g):
    """n unit vectors uniform in the footprint (octant, sphere, or a cap at 40, 30 degrees)."""
    u, v = _rand(g, n), _rand(g, n)
    if sky == "cap":
        c = torch.tensor([[math.cos(30 * DEG) * math.cos(40 * DEG), math.cos(30 * DEG) * math.sin(40 * DEG),
                           math.sin(30 * DEG)]], dtype=torch.float64, device="cuda")
        e_a, e_d = _tangent(c)
        cs = 1.0 - u * (1.0 - math.cos(radius * DEG))
        sn, pa = torch.sqrt((1.0 - cs * cs).clamp_min(0.0)), 2.0 * math.pi * v
        p = cs[:, None] * c + (sn * torch.cos(pa))[:, None] * e_a + (sn * torch.sin(pa))[:, None] * e_d
        return _unit(p)
    z, ra = (u, v * 0.5 * math.pi) if sky == "octant" else (2.0 * u - 1.0, v * 2.0 * math.pi)
    rho = torch.sqrt((1.0 - z * z).clamp_min(0.0))
    return _unit(torch.stack([rho * torch.cos(ra), rho * torch.sin(ra), z], 1))


def _unit(p):
    return (p / torch.sqrt((p * p).sum(1, keepdim=True))).contiguous()


def _clustered(n, clusters, sigma, sky, radius, g):
    """70% of n points in Gaussian clusters (tangent plane), 30% uniform, in random order."""
    m = int(round(0.7 * n))
    c = _uniform(clusters, sky, radius, g)[torch.randint(clusters, (m,), generator=g, device="cuda")]
    e_a, e_d = _tangent(c)
    off = torch.randn(m, 2, generator=g, device="cuda", dtype=torch.float64) * (sigma * DEG)
    p = _unit(c + off[:, :1] * e_a + off[:, 1:] * e_d)
    if sky == "octant":  # members that fall outside are folded back in
        p = p.abs()
    p = torch.cat([p, _uniform(n - m, sky, radius, g)])
    return p[torch.randperm(n, generator=g, device="cuda")].contiguous()


def _edges(c):
    if c["bins"] == "lin":
        t = np.linspace(c["lo"], c["hi"], c["nb"] + 1) * DEG
    else:
        t = np.geomspace(c["lo"], c["hi"], c["nb"] + 1) * DEG
    return t


def _sky(case, seed, n, k):
    """Catalog k of a case: 0 the data, 1 the randoms."""
    g = _gen(seed, k)
    radius = case.get("radius", 0.0)
    if k == 1:
        return _uniform(n, case["sky"], radius, g)
    return _clustered(n, case.get("clusters", 128), case.get("sigma", 0.5), case["sky"], radius, g)


def _box(case, seed, k):
    g = _gen(seed, k)
    n, side = case["nd"] if k == 0 else case["nr"], case["side"]
    p = _rand(g, n, 3) * side
    if k == 0:
        m = int(round(0.7 * n))
        c = (_rand(g, 4096, 3) * side)[torch.randint(4096, (m,), generator=g, device="cuda")]
        p[:m] = (c + 2.0 * torch.randn(m, 3, generator=g, device="cuda", dtype=torch.float64)).clamp(0.0, side)
        p = p[torch.randperm(n, generator=g, device="cuda")]
    return p.contiguous()


def _patches(case, seed):
    """Data and twice as many randoms, cut into compact sky patches of lognormal sizes."""
    nd, npatch = case["nd"], case["patches"]
    sizes = np.random.default_rng(seed).lognormal(0.0, 1.0, npatch).clip(0.2, 30.0)
    cut = np.concatenate([[0.0], np.cumsum(sizes)])
    off = np.round(cut / cut[-1] * nd).astype(np.int64)
    sky = {"sky": "octant", "clusters": 1024, "sigma": 0.2}
    out = []
    for k, n in ((0, nd), (1, 2 * nd)):
        p = _sky(sky, seed, n, k)
        band = (torch.asin(p[:, 2].clamp(-1, 1)) / (0.5 * math.pi) * 23).long().clamp(max=22).double()
        out.append(p[torch.argsort(band * 10.0 + torch.atan2(p[:, 1], p[:, 0]))].contiguous())
    return out[0], out[1], off, 2 * off


def _jobs(case, seed):
    """The burst's jobs: (data, randoms, edges) as host arrays, sizes log-uniform.

    The sizes are the case's (spread evenly over the logarithm); the seed makes the points."""
    jobs = []
    for k in range(case["jobs"]):
        f = (k * 0.6180339887498949 + 0.31) % 1.0
        n = int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** f))
        c = {"sky": "cap", "radius": 5.0 + 25.0 * ((k * 0.414) % 1.0)}
        d, r = _sky(c, seed * 64 + k, n, 0), _sky(c, seed * 64 + k, 2 * n, 1)
        jobs.append((d.cpu().numpy(), r.cpu().numpy(), np.linspace(0.0, 2.0, 21 + (k * 17) % 61) * DEG))
    return jobs


# ------------------------------------------------------------------ one pass
_MODE = {"screen": {}, "prune": {"flags": tpcf.TPCF_F_PRUNE}, "plain": {"precision": tpcf.TPCF_PLAIN_FP64},
         "check": {"flags": tpcf.TPCF_F_CHECK_OVERFLOW}}


def prepare(case, seed):
    """A program's context and what it keeps there: catalogs, bins, a captured graph; or its host arrays."""
    op = case["op"]
    st = {"case": case, "ctx": tpcf.Context(device=0, **_MODE[case.get("mode", "screen")])}
    ctx = st["ctx"]
    stream = torch.cuda.current_stream()
    if op == "correlate":
        st["d"], st["r"] = (_sky(case, seed, n, k).cpu().numpy() for k, n in ((0, case["nd"]), (1, case["nr"])))
        st["edges"] = _edges(case)
    elif op == "serve":
        st["jobs"] = _jobs(case, seed)
    elif op in ("patches", "jackknife"):
        d, r, do, ro = _patches(case, seed)
        st["d"], st["r"] = ctx.catalog(d, stream, do), ctx.catalog(r, stream, ro)
        st["bins"] = ctx.bins(_edges(case))
    elif op == "box":
        st["d"], st["r"] = ctx.catalog3d(_box(case, seed, 0), stream), ctx.catalog3d(_box(case, seed, 1), stream)
        st["bins"] = ctx.bins3d(np.geomspace(case["lo"], case["hi"], case["nb"] + 1))
    else:
        st["d"] = ctx.catalog(_sky(case, seed, case["nd"], 0), stream)
        if op == "count" and case["part"] != "auto":
            st["r"] = ctx.catalog(_sky(case, seed, case["nr"], 1), stream)
        st["bins"] = ctx.bins(_edges(case))
        if op == "graph":
            st["graph"] = ctx.graph(tpcf.TPCF_GRAPH_AUTO, st["d"], None, st["bins"])
    return st


def run(st):
    """One pass; counting calls on resident catalogs leave their histograms on the device."""
    case, ctx = st["case"], st["ctx"]
    op = case["op"]
    if op == "correlate":
        return ctx.correlate(st["d"], st["r"], st["edges"])
    if op == "serve":
        ids = [ctx.submit(d, r, e) for d, r, e in st["jobs"]]
        res = [ctx.poll(i, len(e)) for i, (_, _, e) in zip(ids, st["jobs"])]
        return [[x["dd"], x["dr"], x["rr"], x["w"]] for x in res]
    stream = torch.cuda.current_stream()
    if op == "graph":
        st["graph"].launch(stream)
        return st["graph"].out
    if op == "patches":
        return ctx.count_patches(st["d"], st["r"], st["bins"], stream, device_out=True)
    if op == "jackknife":
        return ctx.jackknife(st["d"], st["r"], st["bins"], stream)
    if op == "count" and case["part"] == "auto":
        return ctx.count_auto(st["d"], st["bins"], stream, device_out=True)
    if op == "count" and case["part"] == "cross":
        return ctx.count_cross(st["d"], st["r"], st["bins"], stream, device_out=True)
    return ctx.count_all(st["d"], st["r"], st["bins"], stream, device_out=True)


# ------------------------------------------------------------------ what a pass cannot do without
def _pairs(nd, nr):
    return nd * (nd - 1) // 2 + nr * (nr - 1) // 2 + nd * nr


def work(case):
    """Bytes: the points (three doubles) and the histograms.  Operations: three multiply-adds for
    each pair counted by brute force (3-D: three differences more); with pruning, for each pair
    of a uniform sky that is in range."""
    op = case["op"]
    if op == "serve":
        n = [int(round(case["nmin"] * (case["nmax"] / case["nmin"]) ** ((k * 0.6180339887498949 + 0.31) % 1.0)))
             for k in range(case["jobs"])]
        return {"bytes": sum(72 * x for x in n), "flops": 6.0 * sum(_pairs(x, 2 * x) for x in n)}
    nd = case["nd"]
    nr = case.get("nr", 0)
    hist = 8 * (case["nb"] + 2)
    if op in ("patches", "jackknife"):
        nr, p = 2 * nd, case["patches"]
        pairs = _pairs(nd, nr) if op == "jackknife" else _pairs(nd // p, nr // p) * p
        return {"bytes": 24 * (nd + nr) + 3 * p * hist, "flops": 6.0 * pairs}
    part = "auto" if op == "graph" else case.get("part", "all")
    pairs = {"all": _pairs(nd, nr), "auto": nd * (nd - 1) // 2, "cross": nd * nr}[part]
    pts = nd if part == "auto" else nd + nr
    per = 9.0 if op == "box" else 6.0
    if case.get("mode") == "prune":
        frac = 0.5 * (1.0 - math.cos(case["hi"] * DEG)) * (8.0 if case["sky"] == "octant" else 1.0)
        pairs = pairs * min(1.0, frac)
    return {"bytes": 24 * pts + (3 if part == "all" else 1) * hist, "flops": per * pairs}


# ------------------------------------------------------------------ the same in plain torch, binary64
def _hist64(a, b, edges, box):
    """Histogram [underflow, bins, overflow] of a against b, or of a's pairs i < j when b is None."""
    auto = b is None
    b = a if auto else b
    e = torch.from_numpy(np.ascontiguousarray(edges)).to(a.device)
    h = torch.zeros(len(edges) + 1, dtype=torch.int64, device=a.device)
    step = max(1, (1 << 26) // max(1, len(b)))
    col = torch.arange(len(b), device=a.device)
    for i in range(0, len(a), step):
        p = a[i:i + step]
        lo = i if auto else 0
        q = b[lo:]
        if box:
            s = [p[:, None, k] - q[None, :, k] for k in range(3)]
            t = torch.sqrt(s[0] * s[0] + s[1] * s[1] + s[2] * s[2])
        else:
            t = p[:, None, 0] * q[None, :, 0] + p[:, None, 1] * q[None, :, 1] + p[:, None, 2] * q[None, :, 2]
            t = torch.acos(t.clamp_(-1.0, 1.0))
        k = torch.bucketize(t, e, right=True)
        if auto:
            k = k[col[None, lo:] > col[i:i + step, None]]
        h += torch.bincount(k.flatten(), minlength=len(edges) + 1)
    return h


def _estimate(dd, dr, rr, nd, nr):
    dd, dr, rr = (x.cpu().numpy()[1:-1].astype(np.float64) for x in (dd, dr, rr))
    n_dd, n_dr, n_rr = dd / (nd * (nd - 1) / 2), dr / (nd * nr), rr / (nr * (nr - 1) / 2)
    with np.errstate(all="ignore"):
        return np.where(rr == 0, np.nan, (n_dd - 2.0 * n_dr + n_rr) / n_rr)


_MOST = 6e9  # pairs counted in plain torch


def exact(case, seed):
    op = case["op"]
    if op == "serve":
        out = []
        for d, r, e in _jobs(case, seed):
            if _pairs(len(d), len(r)) > 5e8:
                out.append([None] * 4)
                continue
            d, r = torch.from_numpy(d).cuda(), torch.from_numpy(r).cuda()
            h = [_hist64(d, None, e, False), _hist64(d, r, e, False), _hist64(r, None, e, False)]
            out.append([x.cpu().numpy().astype(np.uint64) for x in h] + [_estimate(*h, len(d), len(r))])
        return out
    if op in ("patches", "jackknife"):
        return None
    nd, nr = case["nd"], case.get("nr", 0)
    part = "auto" if op == "graph" else case.get("part", "all")
    if {"all": _pairs(nd, nr), "auto": nd * nd // 2, "cross": nd * nr}[part] > _MOST:
        return None
    if op == "box":
        d, r, e = _box(case, seed, 0), _box(case, seed, 1), np.geomspace(case["lo"], case["hi"], case["nb"] + 1)
    else:
        d, e = _sky(case, seed, nd, 0), _edges(case)
        r = _sky(case, seed, nr, 1) if part != "auto" else None
    box = op == "box"
    if part == "auto":
        return _hist64(d, None, e, box)
    if part == "cross":
        return _hist64(d, r, e, box)
    h = [_hist64(d, None, e, box), _hist64(d, r, e, box), _hist64(r, None, e, box)]
    if op == "correlate":
        return [x.cpu().numpy().astype(np.uint64) for x in h] + [_estimate(*h, nd, nr)]
    return h
