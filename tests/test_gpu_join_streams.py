"""Joins beside other work: a host-buffer join behind work on its stream, and threads
whose joins need different amounts of shared memory."""
import threading

import numpy as np
import pytest

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


def test_threads_with_different_shared_memory(cuda, sdblib):
    """Two threads' joins through the same kernel, of few polygons and of many."""
    torch = cuda
    rng = np.random.default_rng(3)
    n = 2000
    x, y, a = dev(torch, *(rng.integers(0, 2 ** B, n, dtype=np.uint32) for _ in range(3)))
    jobs, fails = [], []
    for P in (8, 1900):
        T = W.voronoi_tiling(rng, P, B, nverts=(4, 8))
        c = sdblib.build_covering(T, B, EPS)
        sdblib.covering_build_table(c, 18)
        want = i64(torch, P), i64(torch, P)
        sdblib.join_aggregate(x, y, a, c, sdblib.LOOKUP_TABLE, *want)
        jobs.append((c, want, (i64(torch, P), i64(torch, P)), torch.cuda.Stream()))
    torch.cuda.synchronize()
    start = threading.Barrier(2)

    def work(c, want, got, stream):
        try:
            start.wait()
            for _ in range(4000):
                sdblib.join_aggregate(x, y, a, c, sdblib.LOOKUP_TABLE, *got, stream=stream)
            stream.synchronize()
            assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        except Exception as e:  # noqa: BLE001
            fails.append(e)
    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not fails, fails
    for j in jobs:
        j[0].free()
