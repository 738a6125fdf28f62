"""Joins at the edges of their dispatch and of their 32-bit counters: the range join on
both sides of the polygon counts that take another kernel, with sums and without; many
points of one polygon whose attributes' low halves are all ones."""
import numpy as np
import pytest

from paper_2010_12548_gb300 import workloads as W

pytestmark = pytest.mark.gpu
B, EPS = 18, 64


def dev(torch, *arrays):
    return [torch.from_numpy(np.ascontiguousarray(v).view(np.int32)).cuda() for v in arrays]


def i64(torch, *shape):
    return torch.full(shape, 7, dtype=torch.int64, device="cuda")


def covering(sdb, T, flags=0, bits=18):
    c = sdb.build_covering(T, B, EPS, flags=flags)
    sdb.covering_build_table(c, bits)
    return c


@pytest.mark.parametrize("P", [255, 300, 301, 650, 800, 801, 1024, 1025])
def test_range_join_by_polygon_count(cuda, sdblib, orc, P):
    torch = cuda
    T = W.voronoi_tiling(np.random.default_rng(P), P, B, nverts=(4, 12))
    rng = np.random.default_rng(1)
    n = 50_003
    x, y = (rng.integers(0, 2 ** B + 50, n, dtype=np.uint32) for _ in range(2))
    a = rng.integers(-2 ** 31, 2 ** 31, n).astype(np.int32)
    x[:9000], y[:9000] = T.x[5], T.y[5]
    want = orc.cover(T, EPS, flagged=True).join_range(x, y, a)
    dx, dy, da = dev(torch, x, y, a)
    c = covering(sdblib, T, sdblib.COVER_BOUNDARY_FLAGS)
    got = [i64(torch, P) for _ in range(5)]  # count, sum, bcount, bsum, babs
    sdblib.join_aggregate_range(dx, dy, da, c, sdblib.LOOKUP_TABLE, got[0], got[2], got[1], got[3],
                                got[4])
    for g, w in zip(got, want):
        assert np.array_equal(g.cpu().numpy(), w.astype(np.int64))
    cnt, bc = i64(torch, P), i64(torch, P)
    sdblib.join_aggregate_range(dx, dy, None, c, sdblib.LOOKUP_TABLE, cnt, bc)
    assert torch.equal(cnt, got[0]) and torch.equal(bc, got[2])
    c.free()


@pytest.mark.parametrize("attr", [0xffff, -1, 0x7fffffff, -2 ** 31])
def test_counters_at_their_ends(cuda, sdblib, orc, attr):
    """24M points at one place: answered by the top level, by the table, and by a search
    of a mixed cell; the counters are flushed several times in every block."""
    torch = cuda
    n = 24_000_001
    T = W.voronoi_tiling(np.random.default_rng(2), 12, B, nverts=(4, 8))
    flat = [sdblib.build_covering(T, B, e) for e in (EPS, 4 * EPS)]
    flagged = covering(sdblib, T, sdblib.COVER_BOUNDARY_FLAGS)
    for c in flat:
        sdblib.covering_build_table(c, 18)
    oc = orc.cover(T, EPS, flagged=True)
    mx, my = int(T.x[0]), int(T.y[0])  # a vertex: a cell of several polygons
    cx, cy = int(T.x[T.ring_off[3]:T.ring_off[4]].mean()), int(T.y[T.ring_off[3]:T.ring_off[4]].mean())
    da = torch.full((n,), attr, dtype=torch.int32, device="cuda")
    for px, py in ((cx, cy), (mx, my), (min(mx + 2 * EPS, 2 ** B - 1), my)):
        dx = torch.full((n,), px, dtype=torch.int32, device="cuda")
        dy = torch.full((n,), py, dtype=torch.int32, device="cuda")
        one = oc.join_range([px], [py], [attr])
        assert one[0].sum() >= 1
        got = [i64(torch, T.n) for _ in range(5)]
        sdblib.join_aggregate_range(dx, dy, da, flagged, sdblib.LOOKUP_TABLE, got[0], got[2],
                                    got[1], got[3], got[4])
        for g, w in zip(got, one):
            assert np.array_equal(g.cpu().numpy(), w.astype(np.int64) * n)
        cnt, sm = i64(torch, 2, T.n), i64(torch, 2, T.n)
        sdblib.join_aggregate_multi(dx, dy, da, flat, sdblib.LOOKUP_TABLE, cnt, sm)
        c1, s1 = i64(torch, 2, T.n), i64(torch, 2, T.n)
        for e in range(2):
            sdblib.join_aggregate(dx, dy, da, flat[e], sdblib.LOOKUP_TABLE, c1[e], s1[e])
        assert torch.equal(cnt, c1) and torch.equal(sm, s1)
        assert np.array_equal(cnt[0].cpu().numpy(), one[0].astype(np.int64) * n)
        assert np.array_equal(sm[0].cpu().numpy(), one[1].astype(np.int64) * n)
    for c in flat + [flagged]:
        c.free()
