"""The resident point set's coordinates come back from the sorted curve ids and
its attributes travel with the sort: viewport queries over the resident points
must equal the plain join over the points as given, for every grid size class
(levels 0, 1 and 2 modulo the three of a table step), at vector remainders,
with duplicates, unaligned inputs and without attributes."""
import numpy as np
import pytest

from paper_2010_12548_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [2, 3, 4, 15, 16, 17, 28, 29, 30])
def test_resident_points_equal_the_points_given(cuda, sdblib, B):
    torch = cuda
    G = 2 ** B
    q = max(1, G // 4)
    # a triangle, a square and an overlapping square
    rings = [[(0, 0), (G - 1, 0), (0, G - 1)], [(0, 0), (2 * q, 0), (2 * q, 2 * q), (0, 2 * q)],
             [(q, q), (G - 1, q), (G - 1, G - 1), (q, G - 1)]]
    off = np.cumsum([0] + [len(r) for r in rings]).astype(np.uint32)
    P = W.Polygons(off, np.array([p[0] for r in rings for p in r], np.uint32),
                   np.array([p[1] for r in rings for p in r], np.uint32), B)
    eps = max(2, G // 64)
    rng = np.random.default_rng(B)
    cov = sdblib.build_covering(P, B, eps)
    for n in (1, 2, 3, 4, 5, 1023, 4097, 20_003):
        for offset in (0, 1):
            x, y = (rng.integers(0, G, n + offset) for _ in range(2))
            x[n // 2:] = x[0]  # duplicates
            a = rng.integers(-2 ** 31, 2 ** 31, n + offset)
            x, y, a = (torch.from_numpy(v.astype(np.int32)).cuda()[offset:] for v in (x, y, a))
            for attr in (a, None):
                want = torch.zeros((2, 3), dtype=torch.int64, device="cuda")
                sdblib.join_aggregate(x, y, attr if attr is not None else torch.zeros_like(x), cov,
                                      sdblib.LOOKUP_BINARY, want[0], want[1])
                p = sdblib.points_create(x, y, attr, B)
                got = torch.zeros((2, 3), dtype=torch.int64, device="cuda")
                for j in range(3):  # polygons overlap: one query each
                    b = sdblib.batch_create(p, P, [(0, 0, G, G, eps, 0, 1)],
                                            np.array([j], np.uint32))
                    sdblib.batch_run(b, sdblib.BATCH_PERSISTENT, got[0, j:j + 1], got[1, j:j + 1])
                    torch.cuda.synchronize()
                    b.free()
                assert torch.equal(got, want), (n, offset, attr is None)
                sdblib.points_build_index(p, 8, 4)
                sdblib.points_aggregate(p, cov, sdblib.LOOKUP_RADIX_SPLINE, got[0], got[1])
                assert torch.equal(got, want), (n, offset, attr is None)
                p.free()
