"""Coverings of few ranges: point-index aggregation where a warp takes 3, 7, 15 or 31
ranges, and learned indexes with more leaves than ranges."""
import numpy as np
import pytest

from paper_2010_12548_gb300 import workloads as W

pytestmark = pytest.mark.gpu
B = 16


def dev(torch, *arrays):
    return [torch.from_numpy(np.ascontiguousarray(v).view(np.int32)).cuda() for v in arrays]


def points(n):
    rng = np.random.default_rng(n)
    return (rng.integers(0, 2 ** B, n, dtype=np.uint32), rng.integers(0, 2 ** B, n, dtype=np.uint32),
            rng.integers(-2 ** 31, 2 ** 31, n).astype(np.int32))


@pytest.mark.parametrize("stars", [False, True])
@pytest.mark.parametrize("eps", [2 ** 17, 725, 182, 91, 46, 23])  # 1 to 119,000 ranges
def test_point_index(cuda, sdblib, orc, eps, stars):
    torch = cuda
    rng = np.random.default_rng(4)
    T = (W.star_polygons(rng, 60, B, radius=(2 ** 11, 2 ** 13)) if stars
         else W.voronoi_tiling(rng, 150, B, nverts=(4, 16)))
    pts = points(30_011)
    p = sdblib.points_create(*dev(torch, *pts), B)
    sdblib.points_build_index(p, 18, 16)
    want = orc.cover(T, eps).point_index_aggregate(*pts)
    c = sdblib.build_covering(T, B, eps)
    for lookup in (sdblib.LOOKUP_BINARY, sdblib.LOOKUP_RADIX_SPLINE):
        cnt, sm = (torch.full((T.n,), 7, dtype=torch.int64, device="cuda") for _ in range(2))
        sdblib.points_aggregate(p, c, lookup, cnt, sm)
        assert np.array_equal(cnt.cpu().numpy().view(np.uint64), want[0])
        assert np.array_equal(sm.cpu().numpy(), want[1])
    c.free()


@pytest.mark.parametrize("leaf_bits,root_bits", [(16, 0), (17, 0), (17, 10), (20, 0), (20, 12)])
@pytest.mark.parametrize("eps", [2 ** 17, 4096, 182, 23])
def test_learned_index_with_more_leaves_than_ranges(cuda, sdblib, orc, eps, leaf_bits, root_bits):
    torch = cuda
    T = W.voronoi_tiling(np.random.default_rng(4), 150, B, nverts=(4, 16))
    pts = points(20_003)
    want = orc.cover(T, eps).join(*pts)
    c = sdblib.build_covering(T, B, eps)
    sdblib.covering_build_index(c, leaf_bits, root_bits=root_bits)
    cnt, sm = (torch.full((T.n,), 7, dtype=torch.int64, device="cuda") for _ in range(2))
    sdblib.join_aggregate(*dev(torch, *pts), c, sdblib.LOOKUP_LEARNED, cnt, sm)
    assert np.array_equal(cnt.cpu().numpy().view(np.uint64), want[0])
    assert np.array_equal(sm.cpu().numpy(), want[1]) and sdblib.covering_fallbacks(c) == 0
    c.free()
