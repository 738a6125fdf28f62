"""The raster join without a canvas (points sorted by pixel), which the default
tile size takes when the canvas is much larger than the point set: equal to the
definitional join and to the canvas at block and tile remainders, with points
outside the grid, and with every point in the canvas's last pixel."""
import numpy as np
import pytest

from paper_2010_12548_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def dev(torch, a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.int32)).cuda()


def points(rng, n, B, where):
    G = 2 ** B
    x, y = (rng.integers(0, G, n, dtype=np.uint32) for _ in range(2))
    if where == "outside":
        x[::3] = G
        y[1::5] = 2 ** 32 - 1
    elif where == "last pixel":
        x[:] = y[:] = G - 1
        x[::2] = G
    a = rng.integers(-2 ** 31, 2 ** 31, n, dtype=np.int64).astype(np.int32)
    return W.Points(x, y, a, B)


@pytest.mark.parametrize("where", ["inside", "outside", "last pixel"])
@pytest.mark.parametrize("n", [0, 1, 255, 257, 4095, 4096, 4097, 20_011])
def test_sorted_pixels_equal_definition_and_canvas(cuda, sdblib, orc, n, where):
    torch = cuda
    B, eps = 16, 3  # 2^15 x 2^15 pixels: more than any n here, several tiles
    rng = np.random.default_rng(n)
    P = W.star_polygons(rng, 7, B, nverts=(3, 20), radius=(2 ** 11, 2 ** 14))
    sq = np.array([0, 2 ** B - 1], np.uint32)  # a square reaching the last pixel
    P = W.Polygons(np.append(P.ring_off, P.ring_off[-1] + 4).astype(np.uint32),
                   np.append(P.x, sq[[0, 1, 1, 0]]), np.append(P.y, sq[[0, 0, 1, 1]]), B)
    pts = points(rng, n, B, where)
    want = orc.join_o2(P, eps, pts)
    x, y, a = dev(torch, pts.x), dev(torch, pts.y), dev(torch, pts.attr)
    for tile_bits in (0, 12):
        for sums in (True, False):
            cnt = torch.full((P.n,), 7, dtype=torch.int64, device="cuda")
            sm = torch.full((P.n,), 7, dtype=torch.int64, device="cuda") if sums else None
            sdblib.raster_join(P, B, eps, x, y, a if sums else None, cnt, sm, tile_bits)
            torch.cuda.synchronize()
            assert np.array_equal(cnt.cpu().numpy().view(np.uint64), want[0]), (tile_bits, sums)
            assert not sums or np.array_equal(sm.cpu().numpy(), want[1]), tile_bits
