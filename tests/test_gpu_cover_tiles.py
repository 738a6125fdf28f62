"""The covering's last five levels as tile bitmaps: entry for entry the oracle's
covering (ranges, lists, raster cells) where the refinement ends in tiles -- at
the shallowest levels that do and at unit cells, with boundary flags, with gaps
between polygons, many polygons in one tile (staged, beyond the stage, and too
many) and polygons that overlap, inside tiles only and over coarser cells."""
import math

import numpy as np
import pytest

from paper_2010_12548_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def polygons(rings, B):
    off = np.cumsum([0] + [len(r) for r in rings]).astype(np.uint32)
    return W.Polygons(off, np.array([p[0] for r in rings for p in r], np.uint32),
                      np.array([p[1] for r in rings for p in r], np.uint32), B)


def eps_of(B, F):
    """The smallest eps whose finest level is F."""
    return max(2, math.isqrt(2 * 4 ** (B - F) - 1) + 1)


def check(sdb, orc, P, B, F, flags):
    eps = eps_of(B, F)
    assert sdb.finest_level(B, eps)[1] == F
    cov = sdb.build_covering(P, B, eps, flags=flags)
    oc = orc.cover(P, eps, flagged=bool(flags))
    st, lo, ids = sdb.covering_export(cov)
    assert np.array_equal(st, oc.start) and np.array_equal(lo, oc.list_off)
    assert np.array_equal(ids, oc.list_ids)
    assert cov.info().n_cells == oc.n_records
    cov.free()
    return oc.n_records


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("B,F,n,drop", [(14, 8, 5, 1), (14, 9, 40, 0), (14, 11, 23, 3), (12, 12, 7, 2),
                                        (16, 13, 60, 2), (28, 10, 30, 1), (30, 9, 12, 5)])
def test_tilings(cuda, sdblib, orc, B, F, n, drop, flags):
    T = W.voronoi_tiling(np.random.default_rng(100 * B + n), n, B, nverts=(4, 24))
    if drop:  # gaps between polygons, at the curve's ends too
        T = T.subset([j for j in range(n) if j % (drop + 1)] or [0])
    check(sdblib, orc, T, B, F, flags)


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("n", [3, 4, 5, 33, 300, 560])
def test_polygons_meeting_in_one_tile(cuda, sdblib, orc, n, flags):
    """n disjoint wedges around the middle of a tile that meets them all (560: more
    than a warp takes), and a square in their middle."""
    B, F = 14, 9
    c, r0, r1 = 2 ** 13 + 512, 450, 7600
    rings = []
    for j in range(n):
        a, b = 2 * math.pi * j / n, 2 * math.pi * (j + 0.6) / n
        rings.append([(c + round(q * math.cos(t)), c + round(q * math.sin(t)))
                      for q, t in ((r0, a), (r1, a), (r1, b), (r0, b))])
    rings.append([(c - 3, c - 3), (c + 3, c - 3), (c + 3, c + 3), (c - 3, c + 3)])
    check(sdblib, orc, polygons(rings, B), B, F, flags)


def test_overlap_inside_tiles_only(cuda, sdblib, orc):
    """Squares that overlap by a few finest cells: apart at the tiles' level."""
    B, F = 14, 12
    s = 4 * 32  # a tile
    rings = []
    for j in range(6):
        x0, y0 = 3 * s * j + 50, 5 * s + 17 * j
        rings.append([(x0, y0), (x0 + 3 * s + 40, y0), (x0 + 3 * s + 40, y0 + 300), (x0, y0 + 300)])
    for flags in (0, 1):
        check(sdblib, orc, polygons(rings, B), B, F, flags)


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("layers", [2, 9, 90, 512, 520])
def test_nested_cells(cuda, sdblib, orc, layers, flags):
    """Polygons over one another: coarse cells of some hold coarse cells and tiles
    of others, up to and beyond the polygons that a thread orders (slots both
    ascending and descending with size), with tiles shared and apart."""
    B, F = 13, 10
    sizes = [400 + 3400 * j // layers for j in range(layers)]
    for order in (sizes, sizes[::-1]):
        rings = [[(4000 - r, 3900 - r), (4011 + r, 3907 - r // 2), (4000 + r, 4100 + r // 2),
                  (3990 - r // 3, 4000 + r)] for r in order]
        check(sdblib, orc, polygons(rings, B), B, F, flags)


@pytest.mark.parametrize("F", [8, 11])
def test_nested_stars(cuda, sdblib, orc, F):
    """Stars with holes anywhere on the grid."""
    B = 13
    S = W.holed_stars(np.random.default_rng(F), 12, B, radius=(2 ** 8, 2 ** 10))
    for flags in (0, 1):
        check(sdblib, orc, S, B, F, flags)


def test_records_and_viewport_clip(cuda, sdblib, orc):
    """Raster cells: a covering alone counts as many as in a batch whose viewport
    is the whole grid, and clipped viewports answer as the definition does."""
    torch = cuda
    B, G = 14, 2 ** 14
    T = W.voronoi_tiling(np.random.default_rng(5), 30, B, nverts=(4, 24))
    rng = np.random.default_rng(6)
    pts = W.Points(rng.integers(0, G, 20_001, dtype=np.uint32),
                   rng.integers(0, G, 20_001, dtype=np.uint32),
                   rng.integers(-1000, 1000, 20_001).astype(np.int32), B)
    x, y, a = (torch.from_numpy(v.view(np.int32)).cuda() for v in (pts.x, pts.y, pts.attr))
    p = sdblib.points_create(x, y, a, B)
    ids = np.arange(T.n, dtype=np.uint32)
    for F in (8, 10, 13):
        eps = eps_of(B, F)
        cells = check(sdblib, orc, T, B, F, 0)
        b = sdblib.batch_create(p, T, [(0, 0, G, G, eps, 0, T.n)], ids)
        assert b.info().n_cells == cells
        b.free()
        views = [(int(x0), int(y0), int(x0 + w), int(y0 + w), eps, 0, T.n)
                 for x0, y0, w in zip(rng.integers(0, G // 2, 9), rng.integers(0, G // 2, 9),
                                      (1, 2, 33, 129, 1000, 4097, 5000, 8191, 8192))]
        b = sdblib.batch_create(p, T, views, ids)
        cnt = torch.zeros(len(views) * T.n, dtype=torch.int64, device="cuda")
        sm = torch.zeros_like(cnt)
        sdblib.batch_run(b, sdblib.BATCH_PERSISTENT, cnt, sm)
        torch.cuda.synchronize()
        for q, v in enumerate(views):
            inside = (pts.x >= v[0]) & (pts.x < v[2]) & (pts.y >= v[1]) & (pts.y < v[3])
            c, s, _ = orc.join_o2(T, eps, pts.take(np.nonzero(inside)[0]))
            assert np.array_equal(cnt[q * T.n:(q + 1) * T.n].cpu().numpy().view(np.uint64), c), v
            assert np.array_equal(sm[q * T.n:(q + 1) * T.n].cpu().numpy(), s), v
        b.free()
