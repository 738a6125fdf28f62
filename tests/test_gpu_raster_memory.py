"""Device memory of the raster join over points sorted by pixel: 24 bytes a point, what a
sort by canvas tile takes (and the canvas besides), not more."""
import subprocess
import sys

import pytest

from paper_2010_12548_gb300 import build

pytestmark = pytest.mark.gpu

CHILD = """
import numpy as np, torch
from paper_2010_12548_gb300 import sdb, workloads as W
n = 40_000_000
x, y = (torch.randint(0, 1 << 24, (n,), dtype=torch.int32, device="cuda") for _ in range(2))
a = torch.ones(n, dtype=torch.int32, device="cuda")
T = W.voronoi_tiling(np.random.default_rng(3), 20, 24, nverts=(4, 12))
cnt = torch.zeros(T.n, dtype=torch.int64, device="cuda")
sm = torch.zeros_like(cnt)
sdb.raster_join(T, 24, 2048, x, y, a, cnt, sm)  # 4^14 pixels: more than one canvas tile
assert torch.equal(cnt, sm) and int(cnt.sum()) >= n
print(sdb.memory_stats()[1])
"""


def test_scratch_per_point(cuda, sdblib):
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=build.ROOT, capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    # 24 bytes, the sort's histograms (1024 bytes per block), rounding to the pool's 32 MB
    assert int(r.stdout) <= 26 * 40_000_000
