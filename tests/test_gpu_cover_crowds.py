"""Many polygons in one tile of a covering: at the edges of what warps and blocks take,
in tiles side by side (the set at a border unchanged), over a coarser cell and at one
place, entry for entry the oracle's covering; and in a time of the order of a few.
Crowds of small polygons are left to the refinement at once."""
import time

import numpy as np
import pytest

from paper_2010_12548_gb300 import workloads as W

pytestmark = pytest.mark.gpu
BITS, EPS = 14, 23  # cells of 16 units, tiles of 512


def polygons(rings):
    off = np.cumsum([0] + [len(r) for r in rings]).astype(np.uint32)
    return W.Polygons(off, np.array([p[0] for r in rings for p in r], np.uint32),
                      np.array([p[1] for r in rings for p in r], np.uint32), BITS)


def box(x, y, w, h):
    return [(x, y), (x + w, y), (x + w, y + h), (x, y + h)]


def squares(n, x0=2060, y0=2060, side=9, pitch=19, cols=25):
    return [box(x0 + pitch * (j % cols), y0 + pitch * (j // cols), side, side) for j in range(n)]


def shuffled(rings, seed=0):
    return [rings[j] for j in np.random.default_rng(seed).permutation(len(rings))]


def check(sdb, orc, rings, flags):
    P = polygons(rings)
    cov = sdb.build_covering(P, BITS, EPS, flags=flags)
    oc = orc.cover(P, EPS, flagged=bool(flags))
    for g, w in zip(sdb.covering_export(cov), (oc.start, oc.list_off, oc.list_ids)):
        assert np.array_equal(g, w)
    assert cov.info().n_cells == oc.n_records
    cov.free()


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("n", [4, 5, 8, 9, 36, 37, 70, 500, 512, 513])
def test_crowds(cuda, sdblib, orc, n, flags):
    check(sdblib, orc, shuffled(squares(n)), flags)
    # bars across tiles side by side: each meets four of them
    bars = [box(2060, 2052 + j * 504 // n, 1900, 9) for j in range(n)]
    check(sdblib, orc, shuffled(bars), flags)


@pytest.mark.parametrize("flags", [0, 1])
@pytest.mark.parametrize("n", [9, 40, 300])
def test_crowds_over_coarser_cells(cuda, sdblib, orc, n, flags):
    """A crowd inside large polygons, whose slots lie before, between and after it."""
    around = [box(1000 - 7 * j, 900, 5000 + 9 * j, 6000) for j in range(12)]
    check(sdblib, orc, shuffled(squares(n) + around), flags)
    bars = [box(2060, 2052 + j * 504 // n, 1900, 9) for j in range(n)]
    check(sdblib, orc, shuffled(bars + around), flags)


@pytest.mark.parametrize("n", [7, 30, 300])
def test_polygons_at_one_place(cuda, sdblib, orc, n):
    """Cells of one place, in no order of their polygons."""
    check(sdblib, orc, shuffled([box(1500, 1700, 3000, 2500)] * n + squares(4, x0=7000)), 0)


def test_a_crowd_takes_no_longer(cuda, sdblib):
    """500 polygons in a tile within 3 times the time of 4 (they took 40 times)."""
    def best(n):
        P, t = polygons(squares(n)), []
        for _ in range(8):
            t0 = time.perf_counter()
            sdblib.build_covering(P, BITS, EPS).free()
            t.append(time.perf_counter() - t0)
        return min(t)
    few = best(4)
    assert best(500) < 3 * few


@pytest.mark.parametrize("n", [257, 1000])
def test_crowds_of_small_polygons_are_built_once(cuda, sdblib, n):
    """Launches of the build, against those of the rule that knows no tiles."""
    P, launched = polygons(squares(n)), []
    for flags in (0, sdblib.COVER_NONCONSERVATIVE):
        before = sdblib.launch_count()
        sdblib.build_covering(P, BITS, EPS, flags=flags).free()
        launched.append(sdblib.launch_count() - before)
    assert launched[0] <= launched[1] + 3
