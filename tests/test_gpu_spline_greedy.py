"""The RadixSpline built by warps must be the exact greedy corridor: its point
count equals a plain integer restatement's, on random, duplicated, regular and
very uneven keys, at the chunk's and the warp's remainders."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
CHUNK = 4096


def curve_ids(x, y, B):
    """Quadrant-digit Hilbert ids (order-1 visit (0,0), (0,1), (1,1), (1,0))."""
    d = np.zeros(len(x), np.uint64)
    sw = np.zeros(len(x), bool)
    cm = np.zeros(len(x), np.int64)
    for lev in range(B - 1, -1, -1):
        xb, yb = (x >> lev) & 1, (y >> lev) & 1
        xt, yt = np.where(sw, yb, xb) ^ cm, np.where(sw, xb, yb) ^ cm
        d = (d << np.uint64(2)) | ((xt << 1) | (xt ^ yt)).astype(np.uint64)
        turn = yt == 0
        sw = np.where(turn, ~sw, sw)
        cm = np.where(turn, cm ^ xt, cm)
    return d


def greedy_points(keys, E):
    """Spline points of the greedy corridor per chunk of 4096 keys, in integers."""
    n, total = len(keys), 0
    for c in range(0, n, CHUNK):
        seg = [(keys[j], j) for j in range(c, min(n, c + CHUNK)) if j == 0 or keys[j] != keys[j - 1]]
        if not seg:
            continue
        total += 1
        base = prev = seg[0]
        up = lo = None  # (rise, run) of the cone's edges from the base
        for k, p in seg[1:]:
            run, rise = k - base[0], p - base[1]
            if up is not None and (up[0] * run < rise * up[1] or rise * lo[1] < lo[0] * run):
                total += 1
                base = prev
                run, rise = k - base[0], p - base[1]
                up = lo = None
            if up is None:
                up, lo = (rise + E, run), (rise - E, run)
            else:
                if (rise + E) * up[1] < up[0] * run:
                    up = (rise + E, run)
                if lo[0] * run < (rise - E) * lo[1]:
                    lo = (rise - E, run)
            prev = (k, p)
        if prev[0] != base[0]:
            total += 1
    return total


def layouts(rng, B, n):
    G = 2 ** B
    yield "uniform", rng.integers(0, G, n), rng.integers(0, G, n)
    yield "lattice", rng.integers(0, 16, n) * (G // 16), rng.integers(0, 16, n) * (G // 16)
    yield "regular", np.arange(n) % min(G, 128), (np.arange(n) // min(G, 128)) % G
    e = rng.integers(0, B, n)
    yield "uneven", (1 << e) - 1 + rng.integers(0, 2, n) * 0, rng.integers(0, 1 << np.maximum(1, e // 2))


@pytest.mark.parametrize("E", [1, 2, 7, 32, 1000])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 4095, 4096, 4097, 12_345])
def test_spline_points_are_the_greedy_ones(cuda, sdblib, n, E):
    torch = cuda
    B = 20
    rng = np.random.default_rng(n + E)
    for name, x, y in layouts(rng, B, n):
        x, y = x.astype(np.int64), y.astype(np.int64)
        keys = [int(k) for k in np.sort(curve_ids(x, y, B))]
        t = [torch.from_numpy(v.astype(np.int32)).cuda() for v in (x, y, np.zeros(n))]
        p = sdblib.points_create(*t, B)
        sdblib.points_build_index(p, 12, E)
        ns, err, _ = sdblib.points_index_stats(p)
        assert ns == greedy_points(keys, E), name
        assert err <= E
        p.free()
