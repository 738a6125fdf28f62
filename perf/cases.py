"""Performance cases: the work that a user of this framework has it do.

Every case is one pass through the Python binding (paper_2010_12548_gb300.sdb),
as a program that holds its inputs and handles calls it.  A case is a dict of
plain values whose "kind" names the path:

  join    points against one covering, COUNT and SUM per polygon
  sweep   points against the coverings of an eps sweep, one pass
  range   the join on a boundary-flagged covering and the result intervals
  host    the join of host arrays (pinned), results on the host
  build   ad-hoc polygons: the sweep's coverings, tables and indexes built, and
          a small set of points joined at every eps
  cover   one covering of a few overlapping polygons with holes, points joined
  raster  the Bounded Raster Join
  ingest  a point set made resident (Hilbert order, prefix sums, spline), then
          one aggregation over it
  query   point-indexed aggregation over resident points
  views   fresh viewport queries: coverings built, joined, dropped
  lod     a prepared batch of viewport queries run again

Point sets follow the workloads' mix (70 % from Gaussian clusters, 30 %
uniform, log-normal fares) or are uniform on the stars' grid; polygons are the
workloads' stars and tilings, the tilings mirrored and transposed by the seed.
"""
import math

import numpy as np
import torch

from paper_2010_12548_gb300 import sdb
from paper_2010_12548_gb300 import workloads as W

LOOKUPS = {"binary": sdb.LOOKUP_BINARY, "learned": sdb.LOOKUP_LEARNED, "table": sdb.LOOKUP_TABLE,
           "table_learned": sdb.LOOKUP_TABLE_LEARNED, "spline": sdb.LOOKUP_RADIX_SPLINE}
STARS_BITS, REGION_BITS, ZONES_BITS, TRACTS_BITS = 16, 20, 24, 28


def listed():
    return [
        # the smallest call: 100k points, 16 overlapping polygons, plain method
        dict(name="join_tiny", kind="join", polys="stars", n=100_000, eps=64, lookup="binary",
             sums=True, offset=0),
        # the headline step at its finest eps: a day's pickups against city zones
        dict(name="join_large", kind="join", polys="zones", n=100_000_000, eps=64,
             lookup="table_learned", sums=True, offset=0),
        # a level-of-detail answer at every eps of the sweep, ragged size
        dict(name="sweep_zones", kind="sweep", n=30_000_001, eps=64, levels=4,
             lookup="table_learned", sums=True),
        # COUNT and SUM with their guaranteed intervals, an ordinary size
        dict(name="range_zones", kind="range", n=10_000_019, eps=256, lookup="table_learned",
             sums=True),
        # a program that holds its points on the host (a loaded file)
        dict(name="host_zones", kind="host", n=20_000_003, eps=64, levels=4,
             lookup="table_learned", sums=True),
        # new polygons: everything from the rings to the first answers
        dict(name="build_zones", kind="build", n=1_000_000, eps=64, levels=4,
             lookup="table_learned", sums=True),
        # a user's few overlapping regions with holes: the general merge, plain join
        dict(name="cover_stars", kind="cover", n=200_000, polygons=64, eps=64, flags=0,
             sums=True),
        # the raster join, the canvas cut into tiles
        dict(name="raster_zones", kind="raster", n=20_000_000, eps=1024, sums=True),
        # a point set arrives and is made resident
        dict(name="ingest_zones", kind="ingest", n=30_000_007, eps=4096, sums=True),
        # census tracts over resident points through the point index
        dict(name="query_tracts", kind="query", n=50_000_000, eps=65536, lookup="spline",
             sums=True),
        # a screenful of new views, each with its own covering
        dict(name="views_tracts", kind="views", n=20_000_000, queries=64, lookup="binary"),
        # the same batch of views asked again as a dashboard refreshes
        dict(name="lod_tracts", kind="lod", n=50_000_000, queries=512, lookup="learned",
             mode="persistent"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["join", "join", "sweep", "range", "host", "build", "cover", "raster",
                       "ingest", "query", "views", "lod"])
    sums = rng.random() < 0.8
    four = ["binary", "learned", "table", "table_learned"]
    if kind == "join":
        if rng.random() < 0.3:
            return dict(kind=kind, polys="stars", n=_log_int(rng, 1_000, 1_000_000),
                        eps=2 ** rng.randint(4, 8), lookup=rng.choice(four), sums=sums,
                        offset=rng.randint(0, 1))
        return dict(kind=kind, polys="zones", n=_log_int(rng, 10_000, 40_000_000),
                    eps=2 ** rng.randint(6, 12), lookup=rng.choice(four), sums=sums,
                    offset=rng.randint(0, 1))
    if kind == "sweep":
        return dict(kind=kind, n=_log_int(rng, 100_000, 30_000_000), eps=2 ** rng.randint(6, 8),
                    levels=rng.randint(2, 4), lookup=rng.choice(four), sums=sums)
    if kind == "range":
        return dict(kind=kind, n=_log_int(rng, 100_000, 20_000_000), eps=2 ** rng.randint(7, 12),
                    lookup=rng.choice(four), sums=sums)
    if kind == "host":
        return dict(kind=kind, n=_log_int(rng, 100_000, 20_000_000), eps=2 ** rng.randint(6, 8),
                    levels=rng.randint(1, 4), lookup=rng.choice(["table", "table_learned"]),
                    sums=sums)
    if kind == "build":
        return dict(kind=kind, n=_log_int(rng, 10_000, 1_000_000), eps=2 ** rng.randint(6, 9),
                    levels=rng.randint(1, 4), lookup=rng.choice(four), sums=sums)
    if kind == "cover":
        return dict(kind=kind, n=_log_int(rng, 1_000, 1_000_000), polygons=_log_int(rng, 4, 64),
                    eps=2 ** rng.randint(6, 9), sums=sums,
                    flags=rng.choice([0, sdb.COVER_BOUNDARY_FLAGS, sdb.COVER_NONCONSERVATIVE]))
    if kind == "raster":
        return dict(kind=kind, n=_log_int(rng, 100_000, 20_000_000), eps=2 ** rng.randint(10, 15),
                    sums=sums)
    if kind == "ingest":
        return dict(kind=kind, n=_log_int(rng, 100_000, 30_000_000), eps=2 ** rng.randint(10, 14),
                    sums=sums)
    if kind == "query":
        return dict(kind=kind, n=_log_int(rng, 1_000_000, 50_000_000),
                    eps=2 ** rng.randint(16, 19), lookup=rng.choice(["spline", "binary"]),
                    sums=sums)
    if kind == "views":
        return dict(kind=kind, n=_log_int(rng, 1_000_000, 20_000_000),
                    queries=_log_int(rng, 1, 64), lookup=rng.choice(["binary", "learned"]))
    return dict(kind=kind, n=_log_int(rng, 1_000_000, 50_000_000), queries=_log_int(rng, 16, 512),
                lookup=rng.choice(["binary", "learned"]),
                mode=rng.choice(["persistent", "graph"]))


# ------------------------------------------------------------------ inputs

def _points(bits, n, seed, clusters=0, sigma=(0, 0), offset=0):
    """x, y, attr int32 CUDA tensors of n points (the workloads' mix, or uniform
    without clusters), starting `offset` elements into their buffers."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    G = 1 << bits
    x, y, a = (torch.empty(n + offset, dtype=torch.int32, device="cuda") for _ in range(3))
    if clusters:
        centre = torch.rand((clusters, 2), generator=g, device="cuda", dtype=torch.float64) * G
        sig = sigma[0] + (sigma[1] - sigma[0]) * torch.rand(clusters, generator=g, device="cuda",
                                                            dtype=torch.float64)
    for lo in range(0, n + offset, 1 << 24):
        m = min(1 << 24, n + offset - lo)
        ux = torch.randint(0, G, (m,), generator=g, device="cuda", dtype=torch.int32)
        uy = torch.randint(0, G, (m,), generator=g, device="cuda", dtype=torch.int32)
        if clusters:
            w = torch.randint(0, clusters, (m,), generator=g, device="cuda")
            z = torch.randn((2, m), generator=g, device="cuda", dtype=torch.float32)
            cx = (centre[w, 0] + z[0] * sig[w]).round_()
            cy = (centre[w, 1] + z[1] * sig[w]).round_()
            use = torch.rand(m, generator=g, device="cuda") < 0.7
            use &= (cx >= 0) & (cx < G) & (cy >= 0) & (cy < G)
            ux = torch.where(use, cx.to(torch.int32), ux)
            uy = torch.where(use, cy.to(torch.int32), uy)
        x[lo:lo + m] = ux
        y[lo:lo + m] = uy
        fare = torch.randn(m, generator=g, device="cuda").mul_(0.8).add_(7.0).exp_()
        a[lo:lo + m] = fare.round_().to(torch.int32)
    return x[offset:], y[offset:], a[offset:]


def _turned(T, turn):
    """The tiling mirrored (bits 0, 1 of turn) and transposed (bit 2), rings
    still counter-clockwise."""
    last = np.uint32((1 << T.grid_bits) - 1)
    x = last - T.x if turn & 1 else T.x
    y = last - T.y if turn & 2 else T.y
    if turn & 4:
        x, y = y, x
    if bin(turn & 7).count("1") & 1:
        off = T.ring_off.astype(np.int64)
        ring = np.repeat(np.arange(T.n), np.diff(off))
        back = off[ring] + off[ring + 1] - 1 - np.arange(len(x))
        x, y = x[back], y[back]
    return W.Polygons(T.ring_off, np.ascontiguousarray(x), np.ascontiguousarray(y), T.grid_bits)


def _stars(seed):
    return W.star_polygons(np.random.default_rng(seed), 16, STARS_BITS)


def _zones(seed):
    return _turned(W.zones263_tiling(), seed % 8)


def _tracts(seed):
    return _turned(W.tracts40k_tiling(), seed % 8)


def _city_points(n, seed, offset=0):
    return _points(ZONES_BITS, n, seed, 32, (2.0 ** 16, 2.0 ** 19), offset)


def _country_points(n, seed):
    return _points(TRACTS_BITS, n, seed, 64, (2.0 ** 20, 2.0 ** 23))


def _viewports(n, seed, polys):
    """n level-of-detail queries as the workload has them (side log-uniform in
    2^14 .. 2^24, eps in 2^6 .. 2^14; the polygons that meet the view first, then
    others), subset sizes a ladder over 1 .. 5000 so that every seed asks for as
    many answers.  Returns (query rows, subset ids)."""
    rng = np.random.default_rng(seed)
    G = 1 << polys.grid_bits
    bb = W.polygon_bboxes(polys).astype(np.int32)
    x0s, y0s, x1s, y1s = (np.ascontiguousarray(bb[:, c]) for c in range(4))
    order = rng.permutation(polys.n)
    sizes = rng.permutation([1 + 4999 * (2 * j + 1) // (2 * n) for j in range(n)])
    rows, ids, off = [], [], 0
    for k in sizes:
        side = int(math.exp(rng.uniform(math.log(2 ** 14), math.log(2 ** 24))))
        x0, y0 = (int(v) for v in rng.integers(0, G - side + 1, size=2))
        meets = (x0s < x0 + side) & (x1s >= x0) & (y0s < y0 + side) & (y1s >= y0)
        turn = np.roll(order, int(rng.integers(0, polys.n)))
        first = meets[turn]
        sub = np.concatenate([turn[first][:k], turn[~first][:max(0, k - int(first.sum()))]])
        rng.shuffle(sub)
        rows.append((x0, y0, x0 + side, y0 + side, 2 ** int(rng.integers(6, 15)), off, k))
        ids.append(sub.astype(np.uint32))
        off += int(k)
    return np.asarray(rows, np.int64), np.concatenate(ids)


def _sweep_eps(case):
    return [case["eps"] << (2 * e) for e in range(case.get("levels", 1) - 1, -1, -1)]


def _lookup_structures(cov, lookup, small=False):
    if lookup in ("table", "table_learned"):
        sdb.covering_build_table(cov, 12 if small else 22)
    if lookup in ("learned", "table_learned"):
        sdb.covering_build_index(cov, 8 if small else 16, root_bits=0)


def _outputs(rows, P, sums):
    shape = (rows, P) if rows else (P,)
    count = torch.empty(shape, dtype=torch.int64, device="cuda")
    return count, torch.empty_like(count) if sums else None


def _point_and_polygon_inputs(case, seed):
    """(polygons, grid bits, (x, y, attr)) of a case."""
    kind = case["kind"]
    if kind == "join" and case["polys"] == "stars":
        return _stars(seed), STARS_BITS, _points(STARS_BITS, case["n"], seed,
                                                 offset=case["offset"])
    if kind == "cover":
        regions = W.holed_stars(np.random.default_rng(seed), case["polygons"], REGION_BITS,
                                radius=(2 ** 14, 2 ** 16))
        return regions, REGION_BITS, _points(REGION_BITS, case["n"], seed)
    if kind in ("query", "views", "lod"):
        return _tracts(seed), TRACTS_BITS, _country_points(case["n"], seed)
    return _zones(seed), ZONES_BITS, _city_points(case["n"], seed, case.get("offset", 0))


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "kind": kind}
    polys, bits, (x, y, a) = _point_and_polygon_inputs(case, seed)
    sums = case.get("sums", True)
    st.update(polys=polys, bits=bits)
    if kind in ("join", "sweep", "range", "host"):
        flags = sdb.COVER_BOUNDARY_FLAGS if kind == "range" else 0
        if "levels" in case:
            covs = sdb.build_coverings(polys, bits, _sweep_eps(case))
        else:
            covs = [sdb.build_covering(polys, bits, case["eps"], flags=flags)]
        for c in covs:
            _lookup_structures(c, case["lookup"], bits == STARS_BITS)
        st.update(covs=covs, lookup=LOOKUPS[case["lookup"]])
    if kind in ("join", "sweep"):
        st["out"] = _outputs(len(st["covs"]) if kind == "sweep" else 0, polys.n, sums)
    elif kind == "range":
        st["out"] = _outputs(0, polys.n, sums)
        st["bout"] = _outputs(0, polys.n, sums)
        st["babs"] = torch.empty_like(st["out"][0]) if sums else None
    elif kind == "host":
        x, y, a = (t.cpu().pin_memory() for t in (x, y, a))
        out = torch.zeros((2, len(st["covs"]), polys.n), dtype=torch.int64).pin_memory()
        st["out"] = (out[0], out[1] if sums else None)
    elif kind in ("raster", "ingest", "build", "cover"):
        st["out"] = _outputs(case.get("levels", 0), polys.n, sums)
        if kind == "ingest":
            st["covs"] = [sdb.build_covering(polys, bits, case["eps"])]
    elif kind == "query":
        st["points"] = sdb.points_create(x, y, a, bits)
        sdb.points_build_index(st["points"])
        st["covs"] = [sdb.build_covering(polys, bits, case["eps"])]
        st["out"] = _outputs(0, polys.n, sums)
        x = y = a = None
    else:  # views, lod
        st["points"] = sdb.points_create(x, y, a, bits)
        queries, ids = _viewports(case["queries"], seed, polys)
        st.update(queries=queries, ids=ids, out=_outputs(0, len(ids), True))
        if kind == "lod":
            b = sdb.batch_create(st["points"], polys, queries, ids)
            sdb.batch_set_lookup(b, LOOKUPS[case["lookup"]])
            st["batch"] = b
            st["stream"] = torch.cuda.Stream() if case["mode"] == "graph" else None
        x = y = a = None
    st.update(x=x, y=y, a=a)
    return st


# ------------------------------------------------------------------ one pass

def run(st):
    kind, case = st["kind"], st["case"]
    x, y, a = st["x"], st["y"], st["a"]
    count, total = st["out"]
    if total is None:
        a = None
    if kind == "join":
        sdb.join_aggregate(x, y, a, st["covs"][0], st["lookup"], count, total)
    elif kind == "sweep":
        sdb.join_aggregate_multi(x, y, a, st["covs"], st["lookup"], count, total)
    elif kind == "range":
        bcount, bsum = st["bout"]
        sdb.join_aggregate_range(x, y, a, st["covs"][0], st["lookup"], count, bcount, total, bsum,
                                 st["babs"])
        bounds = sdb.result_bounds(count, bcount, total, bsum, st["babs"])
        return [t for t in (count, total, bcount, bsum, st["babs"], *bounds) if t is not None]
    elif kind == "host":
        sdb.join_aggregate_host_ptrs(x.data_ptr(), y.data_ptr(),
                                     None if a is None else a.data_ptr(), x.numel(), st["covs"],
                                     st["lookup"], count.data_ptr(),
                                     None if total is None else total.data_ptr())
    elif kind == "build":
        covs = sdb.build_coverings(st["polys"], st["bits"], _sweep_eps(case))
        for e, c in enumerate(covs):
            _lookup_structures(c, case["lookup"])
            sdb.join_aggregate(x, y, a, c, LOOKUPS[case["lookup"]], count[e],
                               None if total is None else total[e])
        sizes = [[i.n_ranges, i.n_list_ids, i.n_cells] for i in (c.info() for c in covs)]
        for c in covs:
            c.free()
        return [count, total if total is not None else count, np.array(sizes, np.int64)]
    elif kind == "cover":
        cov = sdb.build_covering(st["polys"], st["bits"], case["eps"], flags=case["flags"])
        sdb.join_aggregate(x, y, a, cov, sdb.LOOKUP_BINARY, count, total)
        info = cov.info()
        cov.free()
        sizes = np.array([info.n_ranges, info.n_list_ids, info.n_cells], np.int64)
        return [count, total if total is not None else count, sizes]
    elif kind == "raster":
        sdb.raster_join(st["polys"], st["bits"], case["eps"], x, y, a, count, total)
    elif kind == "ingest":
        p = sdb.points_create(x, y, a if a is not None else st["a"], st["bits"])
        sdb.points_build_index(p)
        sdb.points_aggregate(p, st["covs"][0], sdb.LOOKUP_RADIX_SPLINE, count, total)
        p.free()
    elif kind == "query":
        sdb.points_aggregate(st["points"], st["covs"][0], LOOKUPS[case["lookup"]], count, total)
    elif kind == "views":
        b = sdb.batch_create(st["points"], st["polys"], st["queries"], st["ids"])
        if case["lookup"] != "binary":
            sdb.batch_set_lookup(b, LOOKUPS[case["lookup"]])
        sdb.batch_run(b, sdb.BATCH_PERSISTENT, count, total)
        b.free()
    else:  # lod
        mode = sdb.BATCH_GRAPH if case["mode"] == "graph" else sdb.BATCH_PERSISTENT
        sdb.batch_run(st["batch"], mode, count, total, stream=st["stream"])
    return [count] if total is None else [count, total]


# ------------------------------------------------------------------ work

# ranges of the zone tiling's covering at eps: they follow the boundary length
# over the finest cell side (20.5M at eps 2^6)
ZONE_RANGES_EPS = 1.31e9
# the same for the tract tiling (6.7e7 at eps 2^12 on its 2^28 grid)
TRACT_RANGES_EPS = 2.74e11
RANGE_BYTES = 16  # start, list offset, payload


def work(case):
    """Bytes a pass cannot do without: its inputs read once, its outputs written
    once (point coordinates, attributes where sums are asked for, the coverings
    where they are the input or the output, 16 bytes per answer)."""
    kind = case["kind"]
    n = case.get("n", 0)
    point = 12 if case.get("sums", True) else 8
    if kind == "cover":
        # boundary length about 2 pi r a star (its radius 2^15), cells of side eps / 2
        ranges = case["polygons"] * 2 * math.pi * 2 ** 15 / (case["eps"] / 2)
        return {"bytes": point * n + RANGE_BYTES * ranges, "flops": 0.0}
    if kind == "build":
        ranges = sum(ZONE_RANGES_EPS / e for e in _sweep_eps(case))
        return {"bytes": point * n + RANGE_BYTES * ranges, "flops": 0.0}
    if kind == "ingest":
        # read the points; write ids, points and prefix sums in curve order
        return {"bytes": 12.0 * n + (8 + 12 + 8) * n, "flops": 0.0}
    if kind == "query":
        # per range its start and payload, and the prefix sum at its end
        return {"bytes": (12.0 + 8) * TRACT_RANGES_EPS / case["eps"], "flops": 0.0}
    if kind in ("views", "lod"):
        # points in the views: mean area of a side log-uniform in 2^14 .. 2^24
        area = (2.0 ** 48 - 2.0 ** 28) / (2 * math.log(2.0 ** 10)) / 2.0 ** (2 * TRACTS_BITS)
        return {"bytes": 12.0 * n * area * case["queries"] + 16.0 * 2500 * case["queries"],
                "flops": 0.0}
    return {"bytes": float(point * n) + 16 * 263 * case.get("levels", 1), "flops": 0.0}


# ------------------------------------------------------------------ exact

PAIRS_MAX = 4_000_000_000  # (cell, edge) tests of one answer


def _edges(polys, j):
    """ax, ay, bx, by of polygon j's edges, over all of its rings (int64)."""
    rings = getattr(polys, "poly_ring_off", None)
    lo, hi = (j, j + 1) if rings is None else (int(rings[j]), int(rings[j + 1]))
    parts = []
    for r in range(lo, hi):
        a, b = int(polys.ring_off[r]), int(polys.ring_off[r + 1])
        x, y = polys.x[a:b].astype(np.int64), polys.y[a:b].astype(np.int64)
        parts.append((x, y, np.roll(x, -1), np.roll(y, -1)))
    return [np.concatenate(v) for v in zip(*parts)]


def _cell_answer(polys, bits, eps, pts, sums):
    """The method's definition in 64-bit integers: a point counts for a polygon
    when the closed cell of side s (the largest power of two with 2 s^2 <= eps^2)
    that holds it meets the closed polygon.  Returns count, sum, and the same
    over the cells that meet the polygon's boundary with the attributes'
    magnitudes; None when it would take too many tests."""
    k = 0
    while k < bits and 2 << (2 * (k + 1)) <= eps * eps:
        k += 1
    x, y, a = (t.long() for t in pts)
    s = 1 << k
    cells, at = torch.unique(((y >> k) << 32) | (x >> k), return_inverse=True)
    cx, cy = (cells & 0xffffffff) << k, (cells >> 32) << k
    weight = torch.zeros((3, len(cells)), dtype=torch.int64, device=x.device)
    weight[0].index_add_(0, at, torch.ones_like(a))
    weight[1].index_add_(0, at, a)
    weight[2].index_add_(0, at, a.abs())
    if len(cells) * float(len(polys.x)) * 3 / polys.n > PAIRS_MAX:
        return None
    out = torch.zeros((5, polys.n), dtype=torch.int64, device=x.device)
    for j in range(polys.n):
        ax, ay, bx, by = (torch.from_numpy(v).cuda() for v in _edges(polys, j))
        near = ((cx <= ax.max()) & (cx + s >= ax.min()) & (cy <= ay.max()) &
                (cy + s >= ay.min())).nonzero().flatten()
        dx, dy = bx - ax, by - ay
        for part in near.split(max(1, (1 << 26) // len(ax))):
            px, py = cx[part][:, None], cy[part][:, None]
            f = dx * (py - ay) - dy * (px - ax)  # side of the corner against each edge
            lo = f + torch.clamp(-dy * s, max=0) + torch.clamp(dx * s, max=0)
            hi = f + torch.clamp(-dy * s, min=0) + torch.clamp(dx * s, min=0)
            meets = ((lo <= 0) & (hi >= 0) & (torch.minimum(ax, bx) <= px + s) &
                     (torch.maximum(ax, bx) >= px) & (torch.minimum(ay, by) <= py + s) &
                     (torch.maximum(ay, by) >= py))
            touch = meets.any(1)
            crosses = ((ay > py) != (by > py)) & torch.where(by > ay, f > 0, f < 0)
            keep = touch | (crosses.sum(1) % 2 == 1)
            w = weight[:, part]
            out[0, j] += w[0][keep].sum()
            out[1, j] += w[1][keep].sum()
            out[2, j] += w[0][touch].sum()
            out[3, j] += w[1][touch].sum()
            out[4, j] += w[2][touch].sum()
    return out


def exact(case, seed):
    """Answers by the definition where that is affordable."""
    kind = case["kind"]
    if kind in ("query", "views", "lod"):
        return None  # answers over tens of thousands of polygons
    if kind == "cover" and case["flags"] == sdb.COVER_NONCONSERVATIVE:
        return None  # another rule for the boundary cells
    if case["n"] > 1_500_000 and kind != "raster":
        return None
    polys, bits, pts = _point_and_polygon_inputs(case, seed)
    sums = case.get("sums", True)
    rows = []
    for eps in _sweep_eps(case):
        r = _cell_answer(polys, bits, eps, pts, sums)
        if r is None:
            return None
        rows.append(r)
    if kind == "range":
        c, t, bc, bt, ba = rows[0]
        if not sums:
            return [c, bc, c - bc, c]
        return [c, t, bc, bt, ba, c - bc, c, t - (ba + bt) // 2, t + (ba - bt) // 2]
    if "levels" in case:
        count, total = (torch.stack([r[i] for r in rows]) for i in (0, 1))
    else:
        count, total = rows[0][0], rows[0][1]
    if kind == "host":
        count, total = count.cpu(), total.cpu()
    if kind in ("build", "cover"):
        return [count, total if sums else count, None]
    return [count, total] if sums else [count]
