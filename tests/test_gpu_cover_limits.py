"""Coverings whose list entries outnumber their cells: polygons that overlap inside
tiles only.  The limit on the entries (2^32 in the library) is lowered in a build of
its own; a covering beyond it is refused, one below it equals the oracle's."""
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
