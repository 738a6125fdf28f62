"""The one-pass sweep join through the cell tables against the separate joins of its
coverings: polygon counts on both sides of what one block's shared memory
accumulates (with sums and without), tables with and without a top level, one to
four coverings, ragged and unaligned points, attributes at the ends of their type."""
import numpy as np
import pytest

from paper_2010_12548_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,bits", [(1, 18), (263, 18), (263, 10), (1650, 18), (1750, 18),
                                    (5000, 18), (5200, 18), (5200, 10)])
def test_sweep_equals_separate_joins(cuda, sdblib, P, bits):
    torch = cuda
    B = 18
    if P == 1:
        T = W.Polygons(np.array([0, 3], np.uint32), np.array([9, 200_000, 70_000], np.uint32),
                       np.array([5, 30_000, 250_001], np.uint32), B)
    else:
        T = W.voronoi_tiling(np.random.default_rng(P), P, B, nverts=(4, 16))
    covs = sdblib.build_coverings(T, B, [1024, 256, 64, 16])
    for c in covs:
        sdblib.covering_build_table(c, bits)
        sdblib.covering_build_index(c, 8, root_bits=0)
    rng = np.random.default_rng(P + bits)
    n = 70_001
    x, y = (rng.integers(0, 2 ** B + 99, n + 1, dtype=np.uint32) for _ in range(2))
    a = rng.integers(-2 ** 31, 2 ** 31, n + 1).astype(np.int32)
    half = n // 2  # all at one place: the longest runs of one polygon, of one mixed cell
    x[:half], y[:half], a[:half] = T.x[0], T.y[0], -2 ** 31
    x, y, a = (torch.from_numpy(v.view(np.int32)).cuda() for v in (x, y, a))
    for lookup in (sdblib.LOOKUP_TABLE, sdblib.LOOKUP_TABLE_LEARNED):
        one_c = torch.zeros((len(covs), T.n), dtype=torch.int64, device="cuda")
        one_s = torch.zeros_like(one_c)
        for at, m in ((0, n), (1, n), (0, 1), (1, 4097), (0, 0)):
            px, py, pa = x[at:at + m], y[at:at + m], a[at:at + m]
            for e, c in enumerate(covs):
                sdblib.join_aggregate(px, py, pa, c, lookup, one_c[e], one_s[e])
            for E in (1, 2, 3, 4):
                cnt = torch.full((E, T.n), 7, dtype=torch.int64, device="cuda")
                sm = torch.full_like(cnt, 7)
                sdblib.join_aggregate_multi(px, py, pa, covs[4 - E:], lookup, cnt, sm)
                assert torch.equal(cnt, one_c[4 - E:]) and torch.equal(sm, one_s[4 - E:]), (at, m, E)
                cnt.fill_(7)
                sdblib.join_aggregate_multi(px, py, None, covs[4 - E:], lookup, cnt)
                assert torch.equal(cnt, one_c[4 - E:]), (at, m, E)
    for c in covs:
        c.free()


@pytest.mark.parametrize("n", [65_535, 65_537, 2 ** 24 + 65_000])
def test_host_join_of_several_coverings(cuda, sdblib, n):
    """Host-buffer joins of one to five coverings, some sharing a pass and some not
    (one without a top level, a chunk too small for a pass), equal device joins."""
    torch = cuda
    B = 18
    T = W.voronoi_tiling(np.random.default_rng(7), 90, B, nverts=(4, 16))
    covs = sdblib.build_coverings(T, B, [1024, 256, 64, 16])
    covs.append(sdblib.build_covering(T, B, 32))
    for i, c in enumerate(covs):
        sdblib.covering_build_table(c, 10 if i == 4 else 18)
    rng = np.random.default_rng(n)
    x, y = (rng.integers(0, 2 ** B + 99, n, dtype=np.uint32) for _ in range(2))
    a = rng.integers(-2 ** 31, 2 ** 31, n).astype(np.int32)
    dx, dy, da = (torch.from_numpy(v.view(np.int32)).cuda() for v in (x, y, a))
    want_c = torch.zeros((5, T.n), dtype=torch.int64, device="cuda")
    want_s = torch.zeros_like(want_c)
    for e, c in enumerate(covs):
        sdblib.join_aggregate(dx, dy, da, c, sdblib.LOOKUP_TABLE, want_c[e], want_s[e])
    want_c, want_s = want_c.cpu().numpy(), want_s.cpu().numpy()
    for pick in ([0], [1, 2], [3, 1, 0], [0, 1, 2, 3], [0, 1, 2, 3, 3], [4, 2], [0, 1, 2, 3, 4]):
        cnt, sm = sdblib.join_aggregate_host(x, y, a, [covs[i] for i in pick], sdblib.LOOKUP_TABLE)
        assert np.array_equal(np.asarray(cnt).astype(np.int64), want_c[pick]), pick
        assert np.array_equal(np.asarray(sm), want_s[pick]), pick
    for c in covs:
        c.free()
