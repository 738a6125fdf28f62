"""Coverings whose list entries outnumber their cells: polygons that overlap inside
tiles only.  The limit on the entries (2^32 in the library) is lowered in a build of
its own; a covering beyond it is refused, one below it equals the oracle's.  And
batches whose polygons overlap: outside a viewport they are answered, inside refused."""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2010_12548_gb300 import build as B
from paper_2010_12548_gb300 import workloads as W

pytestmark = pytest.mark.gpu
LIMIT = 500_000


def corridors(n, bits=14, cell=4):
    """n corridors of 24 cells (less than a tile) along one track, a few cells apart."""
    rng = np.random.default_rng(1)
    o = rng.integers(-5, 6, n) * cell + np.arange(n) % cell
    x = np.tile(np.array([500, 15000, 15000, 500]), n)
    y = (np.array([3000, 8000, 8000 + 24 * cell, 3000 + 24 * cell]) + o[:, None]).ravel()
    return W.Polygons(4 * np.arange(n + 1, dtype=np.uint32), x.astype(np.uint32),
                      y.astype(np.uint32), bits)


CHILD = """
import sys
import numpy as np
from paper_2010_12548_gb300 import sdb
from tests.test_gpu_cover_limits import corridors
sdb.LIB_PATH = sys.argv[1]
few = sdb.build_covering(corridors(12), 14, 6)
np.savez(sys.argv[2], *sdb.covering_export(few))
try:
    sdb.build_covering(corridors(20), 14, 6)
    print("made")
except sdb.SdbError as e:
    print("status", e.status, e)
"""


def test_list_entries_beyond_the_limit_are_refused(cuda, sdblib, orc, tmp_path):
    many, few = orc.cover(corridors(20), 6), orc.cover(corridors(12), 6)
    assert many.n_records < LIMIT <= len(many.list_ids) and len(few.list_ids) < LIMIT
    obj, so = str(tmp_path / "covertiles.o"), str(tmp_path / "libsdb.so")
    subprocess.check_call([B.nvcc(), *B.ARCH, *B.FLAGS, f"-DSDB_LIST_LIMIT={LIMIT}", "-c",
                           os.path.join(B.CSRC, "covertiles.cu"), "-o", obj])
    objs = [os.path.join(B.BUILD, s.replace(".cu", ".o")) for s in B.SOURCES]
    subprocess.check_call([B.nvcc(), *B.ARCH, "-shared", "-cudart", "static", "-o", so,
                           *[obj if o.endswith("covertiles.o") else o for o in objs]])
    out = str(tmp_path / "few.npz")
    r = subprocess.run([sys.executable, "-c", CHILD, so, out], cwd=B.ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert r.stdout.startswith(f"status {sdblib.SDB_ENOMEM} "), r.stdout
    got = np.load(out)
    for k, w in zip(got.files, (few.start, few.list_off, few.list_ids)):
        assert np.array_equal(got[k], w)


def test_more_entries_than_cells(cuda, sdblib, orc):
    oc = orc.cover(corridors(60), 6)
    assert len(oc.list_ids) > 1.9 * oc.n_records
    cov = sdblib.build_covering(corridors(60), 14, 6)
    for g, w in zip(sdblib.covering_export(cov), (oc.start, oc.list_off, oc.list_ids)):
        assert np.array_equal(g, w)
    cov.free()


def square(x, y, side):
    return [(x, y), (x + side, y), (x + side, y + side), (x, y + side)]


@pytest.mark.parametrize("eps", [64, 32])  # cells of 32 or 16, tiles of 32 x 32 cells
def test_overlap_outside_the_viewport(cuda, sdblib, orc, eps):
    """A small square inside a large one's interior, in a tile that the viewport's edge
    cuts: its cells start just outside the viewport."""
    torch = cuda
    bits = 14
    rings = [square(100, 100, 7900), square(1510, 1510, 60), square(9000, 9000, 700)]
    T = W.Polygons(np.array([0, 4, 8, 12], np.uint32),
                   np.array([p[0] for r in rings for p in r], np.uint32),
                   np.array([p[1] for r in rings for p in r], np.uint32), bits)
    rng = np.random.default_rng(3)
    pts = W.Points(*(rng.integers(1000, 2000, 5000, dtype=np.uint32) for _ in range(2)),
                   rng.integers(-9, 9, 5000).astype(np.int32), bits)
    p = sdblib.points_create(*(torch.from_numpy(v.view(np.int32)).cuda()
                               for v in (pts.x, pts.y, pts.attr)), bits)
    ids = np.arange(3, dtype=np.uint32)
    other = (8900, 8900, 9900, 9900, eps, 0, 3)
    view = (1100, 1100, 1500, 1500, eps, 0, 3)
    b = sdblib.batch_create(p, T, [view, other], ids)
    assert b.info().n_pairs >= 3  # the small square is a candidate of the view
    cnt = torch.zeros(6, dtype=torch.int64, device="cuda")
    sm = torch.zeros_like(cnt)
    sdblib.batch_run(b, sdblib.BATCH_PERSISTENT, cnt, sm)
    inside = (pts.x >= 1100) & (pts.x < 1500) & (pts.y >= 1100) & (pts.y < 1500)
    c, s, _ = orc.join_o2(T, eps, pts.take(np.nonzero(inside)[0]))
    assert c[0] > 0 and np.array_equal(cnt[:3].cpu().numpy().view(np.uint64), c)
    assert np.array_equal(sm[:3].cpu().numpy(), s) and not cnt[3:].any()
    b.free()
    with pytest.raises(sdblib.SdbError, match="overlap"):  # reaches into the small square
        sdblib.batch_create(p, T, [(1100, 1100, 1550, 1550, eps, 0, 3), other], ids)
