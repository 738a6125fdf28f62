"""Batches whose tile setting is much longer than their ranges of points: the work does
not grow with the setting, the results and the reported tiles follow it."""
import numpy as np
import pytest

from paper_2010_12548_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_tiles_longer_than_everything(cuda, sdblib):
    torch = cuda
    B, n = 20, 40_001
    rng = np.random.default_rng(8)
    T = W.voronoi_tiling(rng, 50, B, nverts=(4, 16))
    x, y = (torch.from_numpy(rng.integers(0, 2 ** B, n, dtype=np.uint32).view(np.int32)).cuda()
            for _ in range(2))
    a = torch.from_numpy(rng.integers(-9, 9, n).astype(np.int32)).cuda()
    p = sdblib.points_create(x, y, a, B)
    corner = rng.integers(0, 2 ** B - 2 ** 17, (300, 2))
    views = [(int(u), int(v), int(u) + 2 ** 17, int(v) + 2 ** 17, 2 ** 12, 0, T.n) for u, v in corner]
    b = sdblib.batch_create(p, T, views, np.arange(T.n, dtype=np.uint32))
    cnt = torch.zeros(len(views) * T.n, dtype=torch.int64, device="cuda")
    sm = torch.zeros_like(cnt)
    got = {}
    for tile, ppt in ((4096, 2), (16384, 2), (16385, 4), (10 ** 6, 1), (2 ** 32 - 1, 2)):
        sdblib.batch_set_tuning(b, tile, ppt)
        ms = []
        for mode in (sdblib.BATCH_PERSISTENT, sdblib.BATCH_PER_QUERY):
            for _ in range(3):
                t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                t0.record()
                sdblib.batch_run(b, mode, cnt, sm)
                t1.record()
                torch.cuda.synchronize()
                ms.append(t0.elapsed_time(t1))
            got[tile, mode] = (cnt.cpu(), sm.cpu())
        # 300 views' ranges of at most 40001 points: well below 50 ms, whatever the tile
        assert min(ms[:3]) < 50, (tile, ms)
        i = b.info()
        assert i.tile == tile and i.points_per_thread == ppt
        if tile >= n:  # one tile per range
            assert i.n_tiles == got.setdefault("ranges", i.n_tiles) <= 81 * len(views)
    first = got[4096, sdblib.BATCH_PERSISTENT]
    assert int(first[0].sum()) > 0
    for k, v in got.items():
        if k != "ranges":
            assert torch.equal(v[0], first[0]) and torch.equal(v[1], first[1]), k
    b.free()
