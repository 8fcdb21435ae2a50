"""The workloads whose speed counts, as a user's program runs them.

Each case is one use of the cross-match through its Python entry points: a
whole step (index build, match, join), a match against a resident index, the
further selections over a pair list, the Exact Value match, a batch of
requests and a burst of served requests. Sizes are those of the benchmark's
workloads and of the tests, or lie between them.

``prepare`` draws the catalogues on the GPU: a case stands for one sky, and
the seed turns it about its poles and shuffles the rows of both catalogues, so
that results are others while their sizes stay (where the turn would change
the regions' orientation on the sky, the rows alone are shuffled). ``run``
makes one pass and returns every output of it, ``exact`` recomputes the numbers in float64
from the definitions with plain torch (a sorted grid over catalogue B and the
azimuthal-equidistant coordinates about each A source).
"""

from __future__ import annotations

import math

import numpy as np
import torch

ARCSEC = math.pi / 648000.0
EQ, GAL = 0, 1
CIRCLE, ELLIPSE, RECT = 0, 1, 2
FP64, FP32 = 0, 1
ALL, BEST = 1, 2
JOINS = ("and", "or", "all1", "all2", "not1_2", "not2_1", "xor")


# ------------------------------------------------------------------ cases

def listed():
    return [
        # A lookup: the sources of one small field against a catalogue that stays on the GPU.
        # Latency and launches are all there is to it.
        dict(name="lookup", kind="match", sky="allsky", n_a=300, n_b=5_000_000, cap_deg=0.5,
             shape=CIRCLE, size=2.0, columns=False, a_frame=EQ, b_frame=GAL, precision=FP32,
             zone=0.0, join="all1", join_selection=BEST),
        # The plain field cross-match, float64 throughout: two catalogues of one square degree.
        dict(name="field_fp64", kind="step", sky="field", n_a=10_000, n_b=10_000, shape=CIRCLE,
             size=1.0, columns=False, a_frame=EQ, b_frame=EQ, precision=FP64, zone=0.0, ids=False,
             join="or", join_selection=ALL),
        # Extended clumps, an ellipse of its own each, against the compact sources of the plane.
        dict(name="clumps", kind="step", sky="plane", n_a=200_000, n_b=5_000_000, shape=ELLIPSE,
             size=60.0, columns=True, a_frame=GAL, b_frame=GAL, precision=FP32, zone=12.0,
             ids=False, join="or", join_selection=ALL),
        # Rectangles (slits, detector footprints) given in equatorial coordinates against a
        # resident galactic catalogue: the rotated, per-source form, at odd sizes.
        dict(name="rects_rotated", kind="match", sky="allsky", n_a=1_500_007, n_b=30_000_001,
             cap_deg=0.0, shape=RECT, size=15.0, columns=True, a_frame=EQ, b_frame=GAL,
             precision=FP32, zone=0.0, join="xor", join_selection=BEST),
        # A mid-sized all-sky survey against another, default partition.
        dict(name="survey", kind="step", sky="allsky", n_a=3_000_017, n_b=12_000_031, shape=CIRCLE,
             size=2.0, columns=False, a_frame=GAL, b_frame=GAL, precision=FP32, zone=0.0, ids=True,
             join="or", join_selection=ALL),
        # The same kind of survey on the all-float64 path.
        dict(name="survey_fp64", kind="step", sky="allsky", n_a=5_000_000, n_b=20_000_000,
             shape=CIRCLE, size=2.0, columns=False, a_frame=GAL, b_frame=GAL, precision=FP64,
             zone=24.0, ids=True, join="or", join_selection=ALL),
        # The largest: all-sky catalogues of 5e7 and 2e8 sources with ids, the whole step.
        dict(name="all_sky", kind="step", sky="allsky", n_a=50_000_000, n_b=200_000_000,
             shape=CIRCLE, size=2.0, columns=False, a_frame=GAL, b_frame=GAL, precision=FP32,
             zone=24.0, ids=True, join="or", join_selection=ALL),
        # Catalogue A matched slice by slice against one resident catalogue of the whole sky.
        dict(name="resident", kind="match", sky="allsky", n_a=10_000_000, n_b=100_000_000,
             cap_deg=0.0, shape=CIRCLE, size=3.0, columns=False, a_frame=GAL, b_frame=GAL,
             precision=FP32, zone=24.0, join="all1", join_selection=ALL),
        # Concentric regions and the further readings of "best pairs" over the clumps' pair list.
        dict(name="clump_levels", kind="levels", sky="plane", n_a=200_000, n_b=5_000_000,
             shape=ELLIPSE, size=60.0, columns=True, a_frame=GAL, b_frame=GAL, precision=FP32,
             zone=12.0, scales=3),
        # Identifiers matched by value.
        dict(name="values", kind="values", n_a=25_000_000, n_b=100_000_000, key="int64",
             join="all1", join_selection=ALL),
        # Uneven requests of every shape, join and size range in one pass over a resident
        # catalogue, all results collected.
        dict(name="batch", kind="batch", n_b=100_000_000, n_req=64, a_lo=1_000, a_hi=4_000_000,
             zone=20.0),
        # A burst of requests to the server, their columns in pinned host memory.
        dict(name="serve", kind="serve", n_b=50_000_000, n_req=24, a_lo=1_000, a_hi=1_000_000,
             zone=20.0),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))))) | 1

    kind = rng.choice(["step"] * 4 + ["match"] * 4 + ["levels", "values", "batch", "serve"])
    if kind == "values":
        n_b = log(10_000, 100_000_000)
        return dict(kind=kind, n_a=max(101, int(n_b * rng.uniform(0.05, 0.3))), n_b=n_b,
                    key=rng.choice(["int64", "float64"]), join=rng.choice(JOINS),
                    join_selection=rng.choice([ALL, BEST]))
    if kind in ("batch", "serve"):
        return dict(kind=kind, n_b=log(1_000_000, 100_000_000 if kind == "batch" else 50_000_000),
                    n_req=rng.randint(3, 64 if kind == "batch" else 24), a_lo=log(100, 2_000),
                    a_hi=log(20_000, 2_000_000 if kind == "batch" else 800_000),
                    zone=rng.choice([0.0, 10.0, 20.0]))
    sky = rng.choice(["field", "plane", "allsky", "allsky"]) if kind != "levels" else "plane"
    if sky == "field":
        n_a = log(100, 100_000)
        n_b = log(1_000, 100_000)
        shape, size, columns = CIRCLE, rng.uniform(0.5, 3.0), False
    elif sky == "plane":
        n_a = log(1_000, 300_000)
        n_b = log(100_000, 6_000_000)
        shape, size, columns = rng.choice([ELLIPSE, RECT]), rng.uniform(10.0, 60.0), True
    else:
        n_b = log(1_000_000, 100_000_000)
        n_a = min(log(300, 20_000_000), n_b // 3)
        shape = rng.choice([CIRCLE, CIRCLE, ELLIPSE, RECT])
        columns = rng.random() < 0.3
        size = rng.uniform(0.5, 5.0) if not columns else rng.uniform(2.0, 15.0)
    precision = rng.choice([FP32, FP32, FP64]) if n_a <= 5_000_000 else FP32
    a_frame, b_frame = rng.choice([(EQ, EQ), (GAL, GAL), (GAL, GAL), (EQ, GAL)])
    if sky == "field":
        a_frame = b_frame = EQ
    if sky == "plane":
        a_frame = b_frame = GAL
    c = dict(kind=kind, sky=sky, n_a=n_a, n_b=n_b, shape=shape, size=size, columns=columns,
             a_frame=a_frame, b_frame=b_frame, precision=precision,
             zone=rng.choice([0.0, 12.0, 24.0]))
    if kind == "levels":
        c.update(scales=rng.randint(1, 6))
    else:
        c.update(join=rng.choice(JOINS), join_selection=rng.choice([ALL, BEST]))
    if kind == "step":
        c.update(ids=rng.random() < 0.5)
    if kind == "match":
        c.update(cap_deg=rng.choice([0.0, 0.5, 5.0]) if sky == "allsky" and n_a < 100_000 else 0.0)
    return c


# ------------------------------------------------------------- catalogues

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _u(g, n, lo=0.0, hi=1.0):
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _log_u(g, n, lo, hi):
    return torch.exp(_u(g, n, math.log(lo), math.log(hi)))


def _destination(lon, lat, dist, bearing):
    """The point at angular distance dist from (lon, lat) at a bearing east of north."""
    lr, br = torch.deg2rad(lon), torch.deg2rad(lat)
    cl, sl, cb, sb = torch.cos(lr), torch.sin(lr), torch.cos(br), torch.sin(br)
    e, n = torch.sin(bearing) * torch.sin(dist), torch.cos(bearing) * torch.sin(dist)
    cd = torch.cos(dist)
    x = cd * cb * cl - e * sl - n * sb * cl
    y = cd * cb * sl + e * cl - n * sb * sl
    z = cd * sb + n * cb
    return (torch.remainder(torch.rad2deg(torch.atan2(y, x)), 360.0),
            torch.rad2deg(torch.atan2(z, torch.hypot(x, y))))


def _moved(g, lon, lat, sigma_arcsec):
    n = lon.numel()
    x = torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * (sigma_arcsec * ARCSEC)
    y = torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * (sigma_arcsec * ARCSEC)
    return _destination(lon, lat, torch.hypot(x, y), torch.atan2(x, y))


def _cap(g, n, lon0, lat0, radius_deg):
    dist = torch.acos(_u(g, n, math.cos(math.radians(radius_deg)), 1.0))
    full = lambda v: torch.full((n,), float(v), dtype=torch.float64, device="cuda")  # noqa: E731
    return _destination(full(lon0), full(lat0), dist, _u(g, n, 0.0, 2 * math.pi))


def _sky(g, sky, n, n_b):
    """n positions: a box of 1e4 sources of B per square degree, the galactic plane strip
    (density falling with |b|), or the whole sky (denser towards the plane)."""
    if sky == "field":
        side = math.sqrt(n_b / 1e4)
        s = _u(g, n, math.sin(math.radians(2.0)), math.sin(math.radians(2.0 + side)))
        return 150.0 + side * _u(g, n), torch.rad2deg(torch.asin(s))
    if sky == "plane":
        b = -0.3 * torch.log1p(-_u(g, n) * (1.0 - math.exp(-1.0 / 0.3)))
        return _u(g, n, 0.0, 60.0), torch.where(_u(g, n) < 0.5, b, -b)
    if sky == "uniform":
        return _u(g, n, 0.0, 360.0), torch.rad2deg(torch.asin(_u(g, n, -1.0, 1.0)))
    grid = torch.linspace(-90.0, 90.0, 1 << 16, device="cuda", dtype=torch.float64)
    dens = (1.0 + 9.0 * torch.exp(-grid.abs() / 10.0)) * torch.cos(torch.deg2rad(grid))
    cdf = torch.cumsum(dens, 0)
    cdf = (cdf - cdf[0]) / (cdf[-1] - cdf[0])
    u = _u(g, n)
    k = torch.searchsorted(cdf, u).clamp_(1, grid.numel() - 1)
    t = (u - cdf[k - 1]) / (cdf[k] - cdf[k - 1])
    return _u(g, n, 0.0, 360.0), grid[k - 1] + t * (grid[k] - grid[k - 1])


def _turn(g, degrees):
    """A longitude shift. Longitudes are kept on a grid of 2^-36 degrees, so that it is exact."""
    return int(torch.randint(0, degrees * 1024, (1,), generator=g, device="cuda")) / 1024.0


def _turned(lon, shift):
    return torch.remainder(torch.round(lon * 2.0 ** 36) * 2.0 ** -36 + shift, 360.0)


def _shuffled(g, *columns):
    perm = torch.randperm(columns[0].numel(), generator=g, device="cuda")
    return [c[perm].contiguous() for c in columns]


def _catalogues(case, g):
    """A and B (in B's frame): 60 % of A (70 % in a field) have a counterpart in B offset by a
    quarter of a small region's size; an all-sky A has sources at both poles and across the
    longitude seam; clumps and compact sources are drawn independently."""
    n_a, n_b, sky = case["n_a"], case["n_b"], case["sky"]
    if case.get("cap_deg"):
        a_lon, a_lat = _cap(g, n_a, 0.2, 40.0, case["cap_deg"])
    else:
        a_lon, a_lat = _sky(g, sky, n_a, n_b)
        if sky == "allsky":
            k = min(10_000, n_a // 50)
            for at, (lon0, lat0) in enumerate(((0.0, 90.0), (0.0, -90.0), (0.0, 20.0))):
                lo, la = _cap(g, k, lon0, lat0, 0.5)
                where = slice(at * k, (at + 1) * k)
                a_lon[where], a_lat[where] = lo, la
    b_lon, b_lat = _sky(g, sky, n_b, n_b)
    if sky != "plane":
        n_c = min(int(n_a * (0.7 if sky == "field" else 0.6)), n_b)
        if n_c:
            pick = torch.randperm(n_a, generator=g, device="cuda")[:n_c]
            lo, la = _moved(g, a_lon[pick], a_lat[pick], 0.25 * min(case["size"], 2.0))
            at = torch.randperm(n_b, generator=g, device="cuda")[:n_c]
            b_lon[at], b_lat[at] = lo, la
    return a_lon, a_lat, b_lon, b_lat


def _region(case, g, n):
    if not case["columns"]:
        r = dict(shape=case["shape"], a=case["size"])
        if case["shape"] != CIRCLE:
            r.update(b=0.6 * case["size"], pa=35.0)
        return r
    a = _log_u(g, n, case["size"] / 12.0, case["size"])
    r = dict(shape=case["shape"], a_col=a)
    if case["shape"] != CIRCLE:
        r.update(b_col=a * _u(g, n, 0.3, 1.0), pa_col=_u(g, n, 0.0, 180.0))
    return r


# galactic <- equatorial: rows are the galactic axes in equatorial coordinates
def _rotation():
    ra, dec, lcp = (math.radians(v) for v in (192.85948, 27.12825, 122.93192))
    z = np.array([math.cos(dec) * math.cos(ra), math.cos(dec) * math.sin(ra), math.sin(dec)])
    n = np.array([-math.sin(dec) * math.cos(ra), -math.sin(dec) * math.sin(ra), math.cos(dec)])
    e = np.array([-math.sin(ra), math.cos(ra), 0.0])
    x = math.cos(lcp) * n + math.sin(lcp) * e
    y = math.sin(lcp) * n - math.cos(lcp) * e
    return np.stack([x, y, z])


def _to_frame(lon, lat, src, dst):
    if src == dst:
        return lon, lat
    m = _rotation() if src == EQ else _rotation().T
    lr, br = torch.deg2rad(lon), torch.deg2rad(lat)
    v = (torch.cos(br) * torch.cos(lr), torch.cos(br) * torch.sin(lr), torch.sin(br))
    x, y, z = (float(r[0]) * v[0] + float(r[1]) * v[1] + float(r[2]) * v[2] for r in m)
    return (torch.remainder(torch.rad2deg(torch.atan2(y, x)), 360.0),
            torch.rad2deg(torch.atan2(z, torch.hypot(x, y))))


def _value_keys(case, seed):
    """90 % of B's keys distinct, 10 % repeats; 60 % of A's keys are keys of B. The seed gives
    other identifiers and another order of the rows."""
    n_a, n_b = case["n_a"], case["n_b"]
    g = _gen(0)
    turn = _gen(seed)
    mult = 0x9E3779B97F4A7C15 - (1 << 64)
    first = int(torch.randint(1, 1 << 40, (1,), generator=turn, device="cuda"))
    n_d = max(1, int(0.9 * n_b))
    ids = torch.arange(n_d + n_a, device="cuda") + first
    if case["key"] == "float64":
        ids = (ids & ((1 << 48) - 1)).to(torch.float64) * 0.125
    else:
        ids = (ids * mult) & ((1 << 63) - 1)
    rep = ids[torch.randint(0, n_d, (n_b - n_d,), generator=g, device="cuda")]
    b = torch.cat([ids[:n_d], rep])
    a = ids[n_d:].clone()
    n_hit = int(0.6 * n_a)
    a[:n_hit] = b[torch.randint(0, n_b, (n_hit,), generator=g, device="cuda")]
    return _shuffled(turn, a)[0], _shuffled(turn, b)[0]


def _requests(case, seed):
    """The resident catalogue and the requests over it: caps of 0.1 to 10 degrees, sizes spread
    evenly over the logarithm of their range, shapes, columns, joins and frames mixed; half of a
    request's sources are offset copies of B sources inside its cap."""
    g = _gen(1)
    h = np.random.Generator(np.random.Philox(key=1))
    served = case["kind"] == "serve"
    b_frame = GAL if served else EQ
    b_lon, b_lat = _sky(g, "allsky" if served else "uniform", case["n_b"], case["n_b"])
    cb = torch.cos(torch.deg2rad(b_lat))
    ub = (cb * torch.cos(torch.deg2rad(b_lon)), cb * torch.sin(torch.deg2rad(b_lon)),
          torch.sin(torch.deg2rad(b_lat)))
    n_req = case["n_req"]
    steps = (h.permutation(n_req) + 0.5) / n_req
    out = []
    for k in range(n_req):
        n_a = int(case["a_lo"] * (case["a_hi"] / case["a_lo"]) ** steps[k])
        rad = 0.5 * float(np.exp(h.uniform(math.log(0.1), math.log(10.0))))
        lon0, lat0 = h.uniform(0.0, 360.0), math.degrees(math.asin(h.uniform(-1.0, 1.0)))
        size = float(np.exp(h.uniform(math.log(0.5), math.log(30.0))))
        frame = int(h.integers(0, 2)) if served else EQ
        lon, lat = _cap(g, n_a, lon0, lat0, rad)
        if frame == b_frame:
            c, s = math.cos(math.radians(lat0)), math.sin(math.radians(lat0))
            dot = (ub[0] * (c * math.cos(math.radians(lon0))) +
                   ub[1] * (c * math.sin(math.radians(lon0))) + ub[2] * s)
            inside = torch.nonzero(dot >= math.cos(math.radians(rad))).flatten()
            if inside.numel():
                m = n_a // 2
                pick = inside[torch.randint(0, inside.numel(), (m,), generator=g, device="cuda")]
                lon[:m], lat[:m] = _moved(g, b_lon[pick], b_lat[pick], 0.3 * size)
        shape = int(h.integers(0, 3))
        region = dict(shape=shape)
        if h.integers(0, 2):
            a = _log_u(g, n_a, 0.5, 30.0)
            region.update(a_col=a, b_col=a * _u(g, n_a, 0.3, 1.0), pa_col=_u(g, n_a, 0.0, 180.0))
        else:
            region.update(a=size, b=size * h.uniform(0.3, 1.0), pa=h.uniform(0.0, 180.0))
        combo = int(h.integers(0, 14))
        out.append(dict(lon=lon, lat=lat, frame=frame, selection=ALL | BEST, join=JOINS[combo % 7],
                        join_selection=ALL if combo < 7 else BEST, **region))
    turn = _gen(seed)
    shift = 0.0 if served else _turn(turn, 360)
    out = [out[k] for k in torch.randperm(n_req, generator=turn, device="cuda").tolist()]
    for q in out:
        q["lon"] = _turned(q["lon"], shift)
        names = [k for k, v in q.items() if isinstance(v, torch.Tensor)]
        q.update(zip(names, _shuffled(turn, *(q[k] for k in names))))
    b_lon, b_lat = _shuffled(turn, _turned(b_lon, shift), b_lat)
    return b_lon, b_lat, b_frame, out


def _inputs(case, seed):
    g = _gen(2)
    a_lon, a_lat, b_lon, b_lat = _catalogues(case, g)
    region = _region(case, g, case["n_a"])
    turn, shift = _gen(seed), 0.0
    if case["a_frame"] == case["b_frame"] or case["shape"] == CIRCLE:
        shift = _turn(turn, {"allsky": 360, "plane": 300, "field": 200}[case["sky"]])
    a_lon, b_lon = _turned(a_lon, shift), _turned(b_lon, shift)
    names = [k for k, v in region.items() if isinstance(v, torch.Tensor)]
    a_lon, a_lat, *cols = _shuffled(turn, a_lon, a_lat, *(region[k] for k in names))
    region.update(zip(names, cols))
    b_lon, b_lat = _shuffled(turn, b_lon, b_lat)
    a_lon, a_lat = _to_frame(a_lon, a_lat, case["b_frame"], case["a_frame"])
    return a_lon.contiguous(), a_lat.contiguous(), b_lon, b_lat, region


# -------------------------------------------------------- prepare and run

def prepare(case, seed):
    from paper_1611_08494_gb300 import xm

    kind = case["kind"]
    if kind == "values":
        a, b = _value_keys(case, seed)
        return dict(case=case, a=a, b=b)
    if kind in ("batch", "serve"):
        b_lon, b_lat, b_frame, reqs = _requests(case, seed)
        index = xm.Index(b_lon, b_lat, frame=b_frame, zone_height_arcsec=case["zone"])
        if kind == "batch":
            return dict(case=case, index=index, reqs=reqs)
        pin = lambda v: v.cpu().pin_memory() if isinstance(v, torch.Tensor) else v  # noqa: E731
        reqs = [{k: pin(v) for k, v in q.items()} for q in reqs]
        return dict(case=case, reqs=reqs, server=xm.Server(index, slots=3, use_graph=True))
    a_lon, a_lat, b_lon, b_lat, region = _inputs(case, seed)
    st = dict(case=case, a_lon=a_lon, a_lat=a_lat, region=region)
    if kind == "step":
        st.update(b_lon=b_lon, b_lat=b_lat, ids=None)
        if case["ids"]:
            st["ids"] = torch.arange(case["n_b"], device="cuda") * 7919 + seed
        return st
    st["index"] = xm.Index(b_lon, b_lat, frame=case["b_frame"], zone_height_arcsec=case["zone"],
                           build_fp64=case["precision"] == FP64)
    if kind == "levels":
        st["result"] = xm.Result(st["index"], a_lon, a_lat, frame=case["a_frame"],
                                 precision=case["precision"], **region)
        st["scales"] = [(k + 1) / (case["scales"] + 1) for k in range(case["scales"])]
    return st


def _outputs(res, rows):
    return dict(a_row=res.a_row, b_row=res.b_row, sep=res.sep, count=res.count, best_b=res.best_b,
                best_sep=res.best_sep, join_a=rows.a_row, join_b=rows.b_row, join_sep=rows.sep)


def _gather(views):
    out = {k: torch.cat([v[k] for v in views]) for k in
           ("a_row", "b_row", "sep", "count", "best_b", "best_sep", "row_a", "row_b", "row_sep")}
    for k in ("n_unmatched_a", "n_unmatched_b"):
        out[k] = np.array([v[k] for v in views], dtype=np.int64)
    return out


def run(state):
    from paper_1611_08494_gb300 import xm

    case, kind = state["case"], state["case"]["kind"]
    if kind == "values":
        res = xm.ValueResult(state["a"], state["b"])
        return _outputs(res, res.join(case["join"], case["join_selection"]))
    if kind == "levels":
        res = state["result"]
        lv, per_b, mutual = res.levels(state["scales"]), res.pick("best_b"), res.pick("mutual")
        out = dict(dist=lv.dist, best_b=lv.best_b, best_dist=lv.best_dist, level=lv.level,
                   n_within=lv.n_within)
        for name, rows in (("per_b", per_b), ("mutual", mutual)):
            out.update({name + "_a": rows.a_row, name + "_b": rows.b_row, name + "_sep": rows.sep})
        return out
    if kind == "batch":
        batch = xm.Batch(state["index"], state["reqs"], use_graph=True)
        return _gather([batch.view(k) for k in range(batch.n)])
    if kind == "serve":
        tickets = [state["server"].submit(**q) for q in state["reqs"]]
        out = _gather([t.wait().view() for t in tickets])
        torch.cuda.current_stream().synchronize()  # before the tickets give their results back
        return out
    index = state.get("index")
    if index is None:
        index = xm.Index(state["b_lon"], state["b_lat"], frame=case["b_frame"], ids=state["ids"],
                         zone_height_arcsec=case["zone"], build_fp64=case["precision"] == FP64,
                         deferred_check=True)
    res = xm.Result(index, state["a_lon"], state["a_lat"], frame=case["a_frame"],
                    precision=case["precision"], **state["region"])
    return _outputs(res, res.join(case["join"], case["join_selection"]))


# ------------------------------------------------------------------- work

def _expected_pairs(case):
    """Members expected: planted counterparts and the chance members of B's density."""
    size, n_a, n_b = case["size"], case["n_a"], case["n_b"]
    mean2 = size * size  # mean of (semi-axis a)^2
    if case["columns"]:
        mean2 = size * size * (1 - 1 / 144.0) / (2 * math.log(12.0))
    ratio = 1.0 if case["shape"] == CIRCLE else 0.65 if case["columns"] else 0.6
    area = mean2 * ratio * (4.0 if case["shape"] == RECT else math.pi) / 3600.0 ** 2
    per_deg2 = {"field": 1e4, "plane": n_b / 60.0 * 1.6, "allsky": n_b / 41253.0 * 1.6}[case["sky"]]
    planted = 0.0 if case["sky"] == "plane" else 0.55 * n_a
    return planted + n_a * area * per_deg2


def work(case):
    """Bytes: every input column once, every output array once. Flops: the region test of every
    member and the unit vectors of every source, as a float32 form takes them."""
    kind = case["kind"]
    if kind == "values":
        n_a, n_b = case["n_a"], case["n_b"]
        pairs = 0.66 * n_a
        rows = _join_rows(case, n_a, n_b, pairs, 0.6 * n_a)
        return dict(bytes=8 * (n_a + n_b) + 20 * n_a + 24 * (pairs + rows), flops=2.0 * (n_a + n_b))
    if kind in ("batch", "serve"):
        lo, hi, n = case["a_lo"], case["a_hi"], case["n_req"]
        n_a = n * (hi - lo) / math.log(hi / lo)
        pairs = 0.5 * n_a
        # A's columns (half of the requests with three region columns), the records of B near
        # them at 16 bytes each, count, best pair, pairs and join rows
        return dict(bytes=n_a * (16 + 12 + 16 + 20) + 24 * (pairs + 0.5 * n_a), flops=60.0 * n_a)
    n_a, n_b = case["n_a"], case["n_b"]
    pairs = _expected_pairs(case)
    columns = 0 if not case["columns"] else 8 if case["shape"] == CIRCLE else 24
    if kind == "levels":
        # A's position and region, both rows and the separation of every pair and B's position;
        # distance, level and the best pairs of both readings
        return dict(bytes=n_a * (16 + columns + 16 + 4 * case["scales"]) + pairs * (24 + 16 + 12) +
                    24 * (min(pairs, n_b) + n_a), flops=60.0 * pairs)
    rows = _join_rows(case, n_a, n_b, pairs, min(pairs, 0.9 * n_a))
    data = n_a * (16 + columns) + n_a * 20 + 24 * (pairs + rows)
    if kind == "step":
        data += n_b * (16 + (8 if case["ids"] else 0))
    else:
        data += 16 * (pairs + n_a)  # of a resident catalogue, what lies near A
    return dict(bytes=data, flops=60.0 * n_a + 12.0 * pairs + (40.0 * n_b if kind == "step" else 0))


def _join_rows(case, n_a, n_b, pairs, matched_a):
    sel = pairs if case["join_selection"] == ALL else matched_a
    un_a, un_b = max(0.0, n_a - matched_a), max(0.0, n_b - min(sel, n_b))
    return {"and": sel, "or": sel + un_a + un_b, "all1": sel + un_a, "all2": sel + un_b,
            "not1_2": un_a, "not2_1": un_b, "xor": un_a + un_b}[case["join"]]


# ------------------------------------------------------------------ exact

class _Grid:
    """Catalogue B sorted by (latitude zone, longitude)."""

    def __init__(self, lon, lat, reach_arcsec):
        self.h = max(reach_arcsec, 20.0) / 3600.0 * 1.0001
        zone = torch.floor((lat + 90.0) / self.h)
        key, self.row = torch.sort(zone * 512.0 + lon)
        self.key = key
        self.lon, self.lat = lon[self.row], lat[self.row]

    def candidates(self, lon, lat, reach_arcsec):
        """(index into A, place in the sorted B) of every B near an A source."""
        reach = reach_arcsec / 3600.0 * 1.000001 + 1e-7
        z0 = torch.floor((lat - reach + 90.0) / self.h)
        z1 = torch.floor((lat + reach + 90.0) / self.h)
        c = torch.cos(torch.deg2rad(lat))
        s = math.sin(math.radians(reach))
        wide = torch.where(lat.abs() + reach >= 90.0 - 1e-6, torch.full_like(c, 360.0),
                           torch.rad2deg(torch.asin((s / c.clamp_min(1e-12)).clamp_max(1.0))) + 1e-7)
        who, lo, hi = [], [], []
        for dz in range(3):
            for turn in (-360.0, 0.0, 360.0):
                a, b = (lon - wide + turn).clamp_min(0.0), (lon + wide + turn).clamp_max(360.0)
                if turn:  # a window of the whole circle is taken once
                    a = torch.where(wide >= 360.0, b, a)
                k = torch.nonzero((a < b) & (z0 + dz <= z1)).flatten()
                if k.numel():
                    base = (z0[k] + dz) * 512.0
                    who.append(k)
                    lo.append(torch.searchsorted(self.key, base + a[k]))
                    hi.append(torch.searchsorted(self.key, base + b[k], right=True))
        who, lo, hi = torch.cat(who), torch.cat(lo), torch.cat(hi)
        n = hi - lo
        first = torch.cumsum(n, 0) - n
        at = torch.repeat_interleave(lo - first, n) + torch.arange(int(n.sum()), device="cuda")
        return torch.repeat_interleave(who, n), at


def _members(grid, lon, lat, region, chunk=1 << 22):
    """a_row, b_row, sep (arcsec) and normalised distance of every member, in ascending order."""
    shape, n = region["shape"], lon.numel()
    full = lambda v: torch.full((n,), float(v), dtype=torch.float64, device="cuda")  # noqa: E731
    a = region["a_col"] if "a_col" in region else full(region["a"])
    b = region["b_col"] if "b_col" in region else full(region.get("b", region.get("a", 0.0)))
    pa = region["pa_col"] if "pa_col" in region else full(region.get("pa", 0.0))
    big = a if shape == CIRCLE else torch.maximum(a, b) if shape == ELLIPSE else torch.hypot(a, b)
    reach = float(big.max()) if n else 0.0
    got = []
    for at in range(0, n, chunk):
        sl = slice(at, min(n, at + chunk))
        who, k = grid.candidates(lon[sl], lat[sl], reach)
        who = who + at
        la, lb = torch.deg2rad(lat[who]), torch.deg2rad(grid.lat[k])
        dl, db = torch.deg2rad(grid.lon[k] - lon[who]), torch.deg2rad(grid.lat[k] - lat[who])
        half = torch.sin(0.5 * dl)
        x = torch.cos(lb) * torch.sin(dl)
        y = torch.sin(db) + 2.0 * torch.cos(lb) * torch.sin(la) * half * half
        z = torch.cos(db) - 2.0 * torch.cos(lb) * torch.cos(la) * half * half
        rho = torch.atan2(torch.hypot(x, y), z) / ARCSEC
        if shape == CIRCLE:
            q = rho / a[who]
        else:
            phi = torch.atan2(x, y) - torch.deg2rad(pa[who])
            u, v = rho * torch.cos(phi) / a[who], rho * torch.sin(phi) / b[who]
            q = torch.hypot(u, v) if shape == ELLIPSE else torch.maximum(u.abs(), v.abs())
        m = q <= 1.0
        got.append((who[m], grid.row[k[m]], rho[m], q[m]))
    who, row, rho, q = (torch.cat(v) for v in zip(*got))
    order = torch.argsort(row, stable=True)
    order = order[torch.argsort(who[order], stable=True)]
    return who[order], row[order], rho[order], q[order]


def _best(who, value):
    """Position of the first smallest value of each A, and A's that have one."""
    order = torch.argsort(value, stable=True)
    order = order[torch.argsort(who[order], stable=True)]
    first = torch.ones(order.numel(), dtype=torch.bool, device="cuda")
    w = who[order]
    first[1:] = w[1:] != w[:-1]
    return order[first]


def _per_a(who, value, n):
    out = torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")
    out[who] = value
    return out


def _join_sep(join, who, row, sep, n_a, n_b):
    """Separations of a join's rows, and the numbers of rows without a partner."""
    has_a = torch.zeros(n_a, dtype=torch.bool, device="cuda")
    has_a[who] = True
    has_b = torch.zeros(n_b, dtype=torch.bool, device="cuda")
    has_b[row] = True
    parts_a, parts_s = [], []
    if join in ("and", "or", "all1", "all2"):
        parts_a.append(who)
        parts_s.append(sep)
    if join in ("or", "all1", "not1_2", "xor"):
        lone = torch.nonzero(~has_a).flatten()
        parts_a.append(lone)
        parts_s.append(torch.full((lone.numel(),), float("nan"), dtype=torch.float64, device="cuda"))
    a_side = torch.zeros(0, dtype=torch.float64, device="cuda")
    if parts_a:
        a_side = torch.cat(parts_s)[torch.argsort(torch.cat(parts_a), stable=True)]
    n_lone_b = int((~has_b).sum()) if join in ("or", "all2", "not2_1", "xor") else 0
    return a_side, n_lone_b


def _exact_pass(grid, n_b, lon, lat, region, join, join_selection):
    n_a = lon.numel()
    who, row, sep, _ = _members(grid, lon, lat, region)
    best = _best(who, sep)
    pick = slice(None) if join_selection == ALL else best
    a_side, lone = _join_sep(join, who[pick], row[pick], sep[pick], n_a, n_b)
    return sep, _per_a(who[best], sep[best], n_a), a_side, lone


def _reach(region):
    a = float(region["a_col"].max()) if "a_col" in region else region["a"]
    return a * (1.5 if region["shape"] == RECT else 1.0)


def exact(case, seed):
    kind = case["kind"]
    if kind == "values":
        return None  # whole numbers, and separations that are zero or missing
    nothing = dict(a_row=None, b_row=None, count=None, best_b=None)
    if kind in ("batch", "serve"):
        b_lon, b_lat, b_frame, reqs = _requests(case, seed)
        grids = {}
        cols = dict(sep=[], best_sep=[], row_sep=[])
        for q in reqs:
            if q["frame"] not in grids:
                grids[q["frame"]] = _Grid(*_to_frame(b_lon, b_lat, b_frame, q["frame"]), 45.0)
            sep, best, rows, _ = _exact_pass(grids[q["frame"]], case["n_b"], q["lon"], q["lat"], q,
                                             q["join"], q["join_selection"])
            for k, v in zip(("sep", "best_sep", "row_sep"), (sep, best, rows)):
                cols[k].append(v)
        return dict(nothing, row_a=None, row_b=None, n_unmatched_a=None, n_unmatched_b=None,
                    **{k: torch.cat(v) for k, v in cols.items()})
    a_lon, a_lat, b_lon, b_lat, region = _inputs(case, seed)
    b_lon, b_lat = _to_frame(b_lon, b_lat, case["b_frame"], case["a_frame"])
    grid = _Grid(b_lon, b_lat, _reach(region))
    if kind == "levels":
        who, row, sep, q = _members(grid, a_lon, a_lat, region)
        best = _best(who, q)
        by_sep = _best(who, sep)
        by_a = torch.argsort(who, stable=True)
        per_b = by_a[_best(row[by_a], sep[by_a])]
        keep = torch.zeros(who.numel(), dtype=torch.bool, device="cuda")
        keep[per_b] = True
        both = torch.zeros_like(keep)
        both[by_sep] = True
        return dict(dist=q, best_b=None, best_dist=_per_a(who[best], q[best], case["n_a"]),
                    level=None, n_within=None, per_b_a=None, per_b_b=None, per_b_sep=sep[keep],
                    mutual_a=None, mutual_b=None, mutual_sep=sep[keep & both])
    sep, best, rows, lone = _exact_pass(grid, case["n_b"], a_lon, a_lat, region, case["join"],
                                        case["join_selection"])
    rows = torch.cat([rows, torch.full((lone,), float("nan"), dtype=torch.float64, device="cuda")])
    return dict(nothing, sep=sep, best_sep=best, join_a=None, join_b=None, join_sep=rows)
