"""Joins beside other work: a host-buffer join behind work on its stream, and threads
whose joins need different amounts of shared memory."""
import os
import subprocess

import numpy as np
import pytest

from paper_2010_12548_gb300 import build
from paper_2010_12548_gb300 import workloads as W

pytestmark = pytest.mark.gpu
B, EPS = 18, 64


def dev(torch, *arrays):
    return [torch.from_numpy(np.ascontiguousarray(v).view(np.int32)).cuda() for v in arrays]


def i64(torch, *shape):
    return torch.full(shape, 7, dtype=torch.int64, device="cuda")


def test_host_join_behind_work_on_its_stream(cuda, sdblib):
    """The host join's copies wait for what was enqueued on the stream before, whose
    scratch its buffers may take over."""
    torch = cuda
    rng = np.random.default_rng(4)
    n = 300_001
    T = W.voronoi_tiling(rng, 60, B, nverts=(4, 12))
    covs = [sdblib.build_covering(T, B, e) for e in (EPS, 4 * EPS)]
    for c in covs:
        sdblib.covering_build_table(c, 18)
    h = [rng.integers(0, 2 ** B, n, dtype=np.uint32) for _ in range(2)]
    h.append(rng.integers(-9, 9, n).astype(np.int32))
    x, y, a = dev(torch, *h)
    want = i64(torch, 2, T.n), i64(torch, 2, T.n)
    sdblib.join_aggregate_multi(x, y, a, covs, sdblib.LOOKUP_TABLE, *want)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    for _ in range(5):
        got = i64(torch, 2, T.n), i64(torch, 2, T.n)
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            torch.cuda._sleep(20_000_000)  # the sweep behind it starts late
        sdblib.join_aggregate_multi(x, y, a, covs, sdblib.LOOKUP_TABLE, *got, stream=s)
        cnt, sm = sdblib.join_aggregate_host(*h, covs, sdblib.LOOKUP_TABLE, stream=s)
        s.synchronize()
        for k in range(2):
            assert torch.equal(got[k], want[k])
        assert np.array_equal(cnt.astype(np.int64), want[0].cpu().numpy())
        assert np.array_equal(sm, want[1].cpu().numpy())
    for c in covs:
        c.free()


THREADS = r"""
#include <cuda_runtime.h>
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "sdb.h"
int main() {
  const uint32_t n = 2000;
  uint32_t* x;
  if (cudaMalloc(&x, n * 4) || cudaMemset(x, 1, n * 4)) return 2;
  sdb_covering* cov[2];
  for (int k = 0; k < 2; ++k) {
    const uint32_t P = k ? 1900 : 8;
    std::vector<uint32_t> off(P + 1), vx, vy;
    for (uint32_t j = 0; j < P; ++j) {
      const uint32_t a = 100 + 300 * (j % 45), b = 100 + 300 * (j / 45);
      for (uint32_t i = 0; i < 4; ++i) {
        vx.push_back(a + (i == 1 || i == 2 ? 200 : 0));
        vy.push_back(b + (i >= 2 ? 200 : 0));
      }
      off[j + 1] = 4 * (j + 1);
    }
    const sdb_polygons p{P, off.data(), vx.data(), vy.data()};
    if (sdb_build_covering(&p, 18, 64, nullptr, &cov[k])) return 3;
    if (sdb_covering_build_table(cov[k], 18, nullptr)) return 4;
  }
  std::atomic<int> failed{0};
  auto work = [&](int k) {
    cudaStream_t s;
    uint64_t* c;
    cudaStreamCreate(&s);
    cudaMalloc(&c, 2 * 1900 * 8);
    for (int i = 0; i < 30000; ++i)
      if (sdb_join_aggregate(x, x, (int32_t*)x, n, cov[k], SDB_LOOKUP_TABLE, c, (int64_t*)c + 1900, s)
          && !failed++)
        printf("%s\n", sdb_last_error());
    cudaStreamSynchronize(s);
  };
  std::thread a(work, 0), b(work, 1);
  a.join();
  b.join();
  printf("failed: %d\n", failed.load());
  return failed != 0;
}
"""


def test_threads_with_different_shared_memory(cuda, sdblib, tmp_path):
    """Two threads' joins through the same kernel, of few polygons and of many."""
    src, exe = tmp_path / "threads.cu", str(tmp_path / "threads")
    src.write_text(THREADS)
    subprocess.check_call([build.nvcc(), *build.ARCH, "-std=c++17", "-I", build.INCLUDE, "-o", exe,
                           str(src), sdblib.LIB_PATH,
                           "-Xlinker", "-rpath=" + os.path.dirname(sdblib.LIB_PATH)])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
