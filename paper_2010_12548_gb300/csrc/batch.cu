// Batched level-of-detail queries over a resident point set.
//
// Users explore data at several levels of detail: an overview first, then
// zooms into regions of interest (Sec. 1, "Motivating Application").  A query
// here is an axis-aligned viewport, a subset of the polygons and a distance
// bound eps; it asks for COUNT and SUM per polygon of the subset over the
// points inside the viewport, answered from the eps-bounded covering (Sec. 2.2,
// Sec. 5.1).
//
//  * Points are made resident once, ordered by their full-resolution Hilbert
//    id, so a viewport is a handful of contiguous index ranges: the viewport is
//    cut into at most 9 x 9 aligned quadtree cells (side <= a quarter of the
//    viewport), each a contiguous id range, found by binary search.
//  * All queries' coverings are built in one level-synchronous pass over the
//    (query, polygon) pairs whose polygon can reach the viewport, cells clipped
//    to the viewport (cover.cu), which keeps them small at fine eps.
//  * The join is one persistent launch: warps stride over small equal units of the
//    (query, point-tile) work items; per unit its two end points are looked up in
//    the query's ranges, per point the viewport test, its id at the query's finest
//    level (a shift of the resident id), a search between the ends' ranges, and
//    per-slot COUNT/SUM in the query's output slice.  Alternatively one launch
//    per query, or the persistent launch replayed as a captured CUDA graph.
//  * Learned lookup (Sec. 3, learned index): each query covering with enough
//    ranges gets a two-level model, a linear root over the span of its range
//    starts (leaf = (h - lo) >> shift) and FP32 linear leaves fitted by least
//    squares with their maximum errors measured by the lookup's own arithmetic;
//    a unit's end points search only their leaf's error window, the result is
//    verified, and binary search over the slice is the counted fallback.
//  * An autotuner picks the tile size and points per thread by timing the
//    candidates on the batch itself.
#include "hilbert.cuh"
#include "sdb_internal.cuh"

#include <algorithm>
#include <cstring>
#include <string>
#include <vector>

namespace sdb {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t NONE = 0xffffffffu;
constexpr int THREADS = 256;
constexpr int MAXC = 81;  // candidate index ranges per query (9 x 9 cells)

using QueryDev = BatchQueryDev;
using ChunkDev = BatchChunkDev;
using TileRec = BatchTile;

// ---------------------------------------------------------------- points
// Four consecutive points per thread (16-byte loads when the arrays allow):
// the id of every point, bound by memory (16 B a point).
__global__ void point_keys_kernel(const uint32_t* __restrict__ x, const uint32_t* __restrict__ y,
                                  uint64_t n, uint32_t B, uint32_t nsteps, uint32_t st0, int vec,
                                  uint64_t* __restrict__ key, unsigned int* __restrict__ bad) {
  __shared__ uint32_t tab[HILBERT3_SMEM_WORDS];
  hilbert3_fill(tab);
  __syncthreads();
  const uint64_t step = (uint64_t)gridDim.x * blockDim.x * 4;
  for (uint64_t i = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4; i < n; i += step) {
    uint32_t xs[4] = {0, 0, 0, 0}, ys[4] = {0, 0, 0, 0};
    if (vec && i + 3 < n) {
      const uint4 xv = __ldg(reinterpret_cast<const uint4*>(x + i));
      const uint4 yv = __ldg(reinterpret_cast<const uint4*>(y + i));
      xs[0] = xv.x; xs[1] = xv.y; xs[2] = xv.z; xs[3] = xv.w;
      ys[0] = yv.x; ys[1] = yv.y; ys[2] = yv.z; ys[3] = yv.w;
    } else {
      for (uint32_t q = 0; q < 4 && i + q < n; ++q) {
        xs[q] = x[i + q];
        ys[q] = y[i + q];
      }
    }
    uint64_t k[4];
    uint32_t any = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      any |= xs[q] | ys[q];
      k[q] = hilbert3_encode(xs[q], ys[q], nsteps, st0, tab);
    }
    if (any >> B) *bad = 1u;
    if (i + 3 < n) {  // key is the library's own array: 16-byte aligned
      *reinterpret_cast<ulonglong2*>(key + i) = make_ulonglong2(k[0], k[1]);
      *reinterpret_cast<ulonglong2*>(key + i + 2) = make_ulonglong2(k[2], k[3]);
    } else {
      for (uint32_t q = 0; q < 4 && i + q < n; ++q) key[i + q] = k[q];
    }
  }
}

// The sorted points' coordinates from their ids (the curve is a bijection at
// the points' own resolution), so the sort carries the attribute itself and
// nothing is gathered: 16 B a point in order instead of three random 32-byte
// sectors (30M points: 1.47 ms of gathers -> 0.16 ms).
__global__ void point_coords_kernel(const uint64_t* __restrict__ key, uint64_t n, uint32_t nsteps,
                                    uint32_t st0, uint32_t* __restrict__ xs,
                                    uint32_t* __restrict__ ys) {
  __shared__ uint32_t tab[HILBERT3_SMEM_WORDS];
  hilbert3_inverse_fill(tab);
  __syncthreads();
  const uint64_t step = (uint64_t)gridDim.x * blockDim.x * 4;
  for (uint64_t i = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) * 4; i < n; i += step) {
    const uint32_t m = (uint32_t)min((uint64_t)4, n - i);
    uint64_t k[4] = {0, 0, 0, 0};
    if (m == 4) {
      const ulonglong2 a = __ldg(reinterpret_cast<const ulonglong2*>(key + i));
      const ulonglong2 b = __ldg(reinterpret_cast<const ulonglong2*>(key + i + 2));
      k[0] = a.x; k[1] = a.y; k[2] = b.x; k[3] = b.y;
    } else {
      for (uint32_t q = 0; q < m; ++q) k[q] = key[i + q];
    }
    uint32_t cx[4], cy[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) hilbert3_decode(k[q], nsteps, st0, tab, &cx[q], &cy[q]);
    if (m == 4) {
      *reinterpret_cast<uint4*>(xs + i) = make_uint4(cx[0], cx[1], cx[2], cx[3]);
      *reinterpret_cast<uint4*>(ys + i) = make_uint4(cy[0], cy[1], cy[2], cy[3]);
    } else {
      for (uint32_t q = 0; q < m; ++q) {
        xs[i + q] = cx[q];
        ys[i + q] = cy[q];
      }
    }
  }
}

// ---------------------------------------------------------------- candidates
// first index in [lo, n) with key >= q
__device__ __forceinline__ uint64_t first_at_least(const uint64_t* __restrict__ key, uint64_t lo,
                                                   uint64_t n, uint64_t q) {
  uint64_t len = n - lo;
  while (len > 0) {
    const uint64_t half = len >> 1;
    if (__ldg(key + lo + half) < q) {
      lo += half + 1;
      len -= half + 1;
    } else {
      len = half;
    }
  }
  return lo;
}

// One block per query: the viewport cut into aligned cells at most a quarter of
// its side (at most 9 x 9), each cell a contiguous id range, turned into point
// index ranges -- one thread per cell, both searches -- then put in order and
// joined where they touch.  The searches are chains of dependent reads: 81 cells
// one after the other in a thread per query took 1.75 ms for 64 queries over 20M
// points, this 37 us.
constexpr int CAND_THREADS = 96;
static_assert(CAND_THREADS >= MAXC, "a thread per cell");
__global__ __launch_bounds__(CAND_THREADS) void candidates_kernel(
    const QueryDev* __restrict__ qd, uint32_t Q, const uint64_t* __restrict__ key, uint64_t n,
    uint32_t B, uint32_t* __restrict__ cand, uint32_t* __restrict__ ncand) {
  __shared__ uint32_t s_a[MAXC], s_b[MAXC], s_oa[MAXC], s_ob[MAXC];
  const uint32_t q = blockIdx.x, t = threadIdx.x;
  const uint32_t x0 = qd[q].x0, y0 = qd[q].y0, x1 = qd[q].x1, y1 = qd[q].y1;
  const uint32_t side = max(x1 - x0, y1 - y0);
  uint32_t lc = 0;  // log2 of the cell side
  while (lc < B && (2u << lc) <= max(1u, side / 4)) ++lc;
  const uint32_t L = B - lc;  // cell level
  const uint32_t cx0 = x0 >> lc, cy0 = y0 >> lc;
  const uint32_t nx = ((x1 - 1) >> lc) - cx0 + 1, ny = ((y1 - 1) >> lc) - cy0 + 1;
  const uint32_t m = min(nx * ny, (uint32_t)MAXC);
  if (t < m) {
    const uint64_t h = hilbert_id(cx0 + t % nx, cy0 + t / nx, L);
    const uint64_t lo = first_at_least(key, 0, n, h << (2 * lc));
    s_a[t] = (uint32_t)lo;
    s_b[t] = (uint32_t)first_at_least(key, lo, n, (h + 1) << (2 * lc));
  }
  __syncthreads();
  if (t < m) {  // cells are disjoint: by start, empty ranges by their place
    uint32_t r = 0;
    for (uint32_t i = 0; i < m; ++i)
      r += s_a[i] < s_a[t] || (s_a[i] == s_a[t] && (s_b[i] < s_b[t] || (s_b[i] == s_b[t] && i < t)));
    s_oa[r] = s_a[t];
    s_ob[r] = s_b[t];
  }
  __syncthreads();
  if (t == 0) {
    uint32_t w = 0;
    uint32_t* out = cand + (size_t)q * MAXC * 2;
    for (uint32_t i = 0; i < m;) {
      uint32_t a = s_oa[i], b = s_ob[i];
      ++i;
      if (a >= b) continue;  // no points
      while (i < m && s_oa[i] <= b) b = max(b, s_ob[i++]);
      out[2 * w] = a;
      out[2 * w + 1] = b;
      ++w;
    }
    ncand[q] = w;
  }
}

// tiles of at most T points per query; over all queries, tiles of at most `asked` points
// (all[0]) and the points of the longest range (all[1])
__global__ void tile_count_kernel(const uint32_t* __restrict__ cand,
                                  const uint32_t* __restrict__ ncand, uint32_t Q, uint32_t T,
                                  uint32_t asked, uint64_t* __restrict__ ntile,
                                  unsigned long long* __restrict__ all) {
  uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= Q) return;
  uint64_t t = 0, ta = 0, most = 0;
  for (uint32_t i = 0; i < ncand[q]; ++i) {
    const uint32_t a = cand[(size_t)q * MAXC * 2 + 2 * i], b = cand[(size_t)q * MAXC * 2 + 2 * i + 1];
    t += ((uint64_t)b - a + T - 1) / T;
    ta += ((uint64_t)b - a + asked - 1) / asked;
    most = max(most, (uint64_t)(b - a));
  }
  ntile[q] = t;
  atomicAdd(all, (unsigned long long)ta);
  atomicMax(all + 1, (unsigned long long)most);
}

// a block per query: one of many points has many tiles
__global__ __launch_bounds__(128) void tile_fill_kernel(const uint32_t* __restrict__ cand,
                                                        const uint32_t* __restrict__ ncand,
                                                        uint32_t T,
                                                        const uint64_t* __restrict__ toff,
                                                        TileRec* __restrict__ tiles) {
  const uint32_t q = blockIdx.x;
  uint64_t t = toff[q];
  for (uint32_t i = 0; i < ncand[q]; ++i) {
    const uint32_t a = cand[(size_t)q * MAXC * 2 + 2 * i], b = cand[(size_t)q * MAXC * 2 + 2 * i + 1];
    const uint64_t m = ((uint64_t)b - a + T - 1) / T;
    for (uint64_t j = threadIdx.x; j < m; j += 128)
      tiles[t + j] = TileRec{q, (uint32_t)(a + j * T), (uint32_t)min((uint64_t)b, a + (j + 1) * T), 0};
    t += m;
  }
}

// ---------------------------------------------------------------- join
struct BatchArgs {
  const uint64_t* key;
  const uint32_t* x;
  const uint32_t* y;
  const int32_t* attr;
  const QueryDev* q;
  const TileRec* tiles;
  const ChunkDev* chunks;
  unsigned long long* count;
  unsigned long long* sum;
  const LeafRec* leaves;          // per-query learned leaves (queries with nleaves > 0)
  unsigned long long* fallbacks;  // learned searches that missed
};

// last r in [0, R) with st[r] <= h (st[R] is the slice's sentinel, above all ids)
__device__ __forceinline__ uint32_t slice_bs(const uint64_t* __restrict__ st, uint32_t R,
                                             uint64_t h) {
  uint32_t lo = 0;
  for (uint32_t len = R + 1; len > 1;) {
    const uint32_t half = len >> 1;
    if (__ldg(st + lo + half) <= h) lo += half;
    len -= half;
  }
  return lo;
}

// the range of id h in a query slice through its learned index: ids outside
// the leaves' span are the first or last range; else the leaf's prediction,
// a search of its error window (an end no probe has proven is read back), and
// binary search over the slice when the window does not bracket h (counted)
__device__ __forceinline__ uint32_t slice_learned(const uint64_t* __restrict__ st,
                                                  const QueryDev& Q, const LeafRec* leaves,
                                                  unsigned long long* fallbacks, uint64_t h) {
  if (h < Q.llo) return 0;
  if (h >= Q.lhi) return Q.R - 1;
  uint64_t l = (h - Q.llo) >> Q.lwshift;
  if (l >= Q.nleaves) l = Q.nleaves - 1;
  uint64_t w0, w1, w2, w3;
  asm("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];"
      : "=l"(w0), "=l"(w1), "=l"(w2), "=l"(w3)
      : "l"(leaves + Q.loff + l));
  LeafRec lr;
  lr.base = w0;
  lr.a = __uint_as_float((uint32_t)w1);
  lr.b = __uint_as_float((uint32_t)(w1 >> 32));
  lr.first = (uint32_t)w2;
  lr.last = (uint32_t)(w2 >> 32);
  lr.errlo = (int32_t)(uint32_t)w3;
  lr.errhi = (int32_t)(uint32_t)(w3 >> 32);
  const int64_t pr = leaf_predict(lr, h);
  int64_t a = pr - lr.errlo, b = pr + lr.errhi;
  if (a < (int64_t)lr.first) a = lr.first;
  if (b > (int64_t)lr.last) b = lr.last;
  if (b < a) b = a;
  uint32_t lo = (uint32_t)a, len = (uint32_t)(b - a + 1), known = 0;
  while (len > 1) {
    const uint32_t half = len >> 1;
    if (__ldg(st + lo + half) <= h) {
      lo += half;
      known |= 1u;
    } else {
      known |= 2u;
    }
    len -= half;
  }
  const bool ok0 = (known & 1u) || __ldg(st + lo) <= h;
  const bool ok1 = (known & 2u) || h < __ldg(st + lo + 1);
  if (ok0 && ok1) return lo;
  atomicAdd(fallbacks, 1ull);
  return slice_bs(st, Q.R, h);
}

// A warp's running total for one output slot, in registers: the points of a work
// unit are in curve order, so whole warps mostly add to the slot they added to
// last, and a slot's total leaves with one atomic pair when another takes over.
struct SlotSum {
  uint32_t slot = NONE;  // all members warp-uniform
  unsigned long long cnt = 0;
  long long sum = 0;
  template <bool SUM>
  __device__ __forceinline__ void flush(const BatchArgs& A, uint32_t lane) {
    if (slot != NONE && lane == 0) {
      atomicAdd(&A.count[slot], cnt);
      if (SUM) atomicAdd(&A.sum[slot], (unsigned long long)sum);
    }
    cnt = 0;
    sum = 0;
  }
};

// A warp takes work units: up to 32 G consecutive points of a (query, tile) work item,
// G to a lane.
// The resident points are in curve order and keep their full-resolution ids, so a
// point's cell id at the query's level is a shift, ids ascend along the unit, and
// only its first and last point are looked up in the whole slice (by the learned
// index or binary search); the others search the few ranges between.  A unit whose
// common quadtree cell lies inside the viewport reads no coordinates.  Points of
// one slot add up across the warp (32-bit reductions of the attribute's halves,
// exact).  A chain of dependent reads bounds it, so units are small and equal and
// many warps work at once (units of 1024 points took 376 us).  Before, every point
// was encoded from its coordinates and looked up by itself, and a block cleared and
// scanned 2048 slots per 4096 points or, for larger subsets, sent two global
// atomics per point: 512 views over 50M points 298 us, this 246 with 4096-point tiles
// and 167 with pieces of 256.
template <int G, bool SUM>
__global__ __launch_bounds__(THREADS) void batch_kernel(BatchArgs A, uint32_t tile_lo,
                                                        uint32_t tile_hi,
                                                        uint32_t units_per_tile) {
  constexpr uint32_t UNIT = 32 * G;
  const uint32_t lane = threadIdx.x & 31;
  SlotSum tot;
  const uint64_t units = (uint64_t)(tile_hi - tile_lo) * units_per_tile;
  const uint64_t step = ((uint64_t)gridDim.x * THREADS) >> 5;
  for (uint64_t u = ((uint64_t)blockIdx.x * THREADS + threadIdx.x) >> 5; u < units; u += step) {
    const TileRec tr = A.tiles[tile_lo + u / units_per_tile];
    const uint64_t b64 = tr.begin + (u % units_per_tile) * UNIT;
    if (b64 >= tr.end) continue;
    // (counted from b: b + UNIT may pass 2^32)
    const uint32_t b = (uint32_t)b64, m = min(tr.end - b, UNIT);
    // the unit's points (past its end: its last point again)
    uint64_t key[G];
#pragma unroll
    for (int g = 0; g < G; ++g) key[g] = __ldg(A.key + b + min(g * 32 + lane, m - 1));
    const QueryDev& Q = A.q[tr.q];
    const ChunkDev C = A.chunks[Q.chunk];
    const uint64_t sbase = Q.sbase;
    const uint64_t* st = C.start + sbase;
    const uint32_t sh = 2 * Q.k;  // finest id at the query's level = key >> sh
    const uint32_t x0 = Q.x0, y0 = Q.y0, x1 = Q.x1, y1 = Q.y1, out = Q.out_off;
    // the smallest quadtree cell that holds all of the unit's points
    const uint64_t first = __shfl_sync(FULL, key[0], 0), last = __shfl_sync(FULL, key[G - 1], 31);
    const uint64_t diff = first ^ last;
    const uint32_t lc = diff ? (64 - __clzll((long long)diff) + 1) / 2 : 0;
    const uint64_t cx = (uint64_t)(__ldg(A.x + b) >> lc) << lc, cy = (uint64_t)(__ldg(A.y + b) >> lc) << lc;
    const bool inside = cx >= x0 && cy >= y0 && cx + (1ull << lc) <= x1 && cy + (1ull << lc) <= y1;
    bool ok[G];
    int32_t av[G];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const uint32_t i = b + g * 32 + lane;
      ok[g] = g * 32 + lane < m;
      av[g] = (SUM && ok[g]) ? __ldg(A.attr + i) : 0;
      if (!inside && ok[g]) {
        const uint32_t x = __ldg(A.x + i), y = __ldg(A.y + i);
        ok[g] = x >= x0 && x < x1 && y >= y0 && y < y1;
      }
    }
    // the ranges of its ends, then of every point between them
    uint32_t r = 0;
    if (lane == 0 || lane == 31) {
      const uint64_t h = (lane ? last : first) >> sh;
      r = Q.nleaves ? slice_learned(st, Q, A.leaves, A.fallbacks, h) : slice_bs(st, Q.R, h);
    }
    const uint32_t lo = __shfl_sync(FULL, r, 0), hi = __shfl_sync(FULL, r, 31);
    uint32_t rr[G];
#pragma unroll
    for (int g = 0; g < G; ++g) rr[g] = lo;
    for (uint32_t len = hi - lo + 1; len > 1;) {
      const uint32_t half = len >> 1;
      uint64_t v[G];
#pragma unroll
      for (int g = 0; g < G; ++g) v[g] = __ldg(st + rr[g] + half);
#pragma unroll
      for (int g = 0; g < G; ++g)
        if (v[g] <= key[g] >> sh) rr[g] += half;
      len -= half;
    }
    uint32_t pay[G];
#pragma unroll
    for (int g = 0; g < G; ++g) pay[g] = ok[g] ? __ldg(C.pay + sbase + rr[g]) : NONE;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const bool list = pay[g] != NONE && pay[g] >= 0x80000000u;
      uint32_t j = 0, j1 = pay[g] != NONE ? 1u : 0u;
      if (list) {
        j = __ldg(C.list_off + (pay[g] & 0x7fffffffu));
        j1 = __ldg(C.list_off + (pay[g] & 0x7fffffffu) + 1);
      }
      for (;;) {  // the points' polygons, one each a round
        uint32_t left = __ballot_sync(FULL, j < j1);
        if (!left) break;
        const uint32_t p = j < j1 ? (list ? __ldg(C.list_ids + j) : pay[g]) : NONE;
        ++j;
        while (left) {
          const uint32_t pl = __shfl_sync(FULL, p, __ffs(left) - 1);
          const bool mine = p == pl;
          const uint32_t group = __ballot_sync(FULL, mine);
          left &= ~group;
          if (out + pl != tot.slot) {
            tot.flush<SUM>(A, lane);
            tot.slot = out + pl;
          }
          tot.cnt += __popc(group);
          if (SUM) {
            const uint32_t l = __reduce_add_sync(FULL, mine ? (uint32_t)av[g] & 0xffffu : 0u);
            const int32_t w = __reduce_add_sync(FULL, mine ? av[g] >> 16 : 0);
            tot.sum += (long long)w * 65536 + (long long)l;
          }
        }
      }
    }
  }
  tot.flush<SUM>(A, lane);
}

// ---------------------------------------------------------------- learned index
// per query with leaves: the span [llo, lhi) of ids between its second range
// start and one past its last range start
__global__ void slice_span_kernel(const QueryDev* __restrict__ qd, uint32_t Q,
                                  const ChunkDev* __restrict__ chunks, uint32_t min_ranges,
                                  uint64_t* __restrict__ span) {
  const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= Q) return;
  const QueryDev d = qd[q];
  if (d.R < 2 || d.R < min_ranges) {
    span[2 * q] = span[2 * q + 1] = 0;
    return;
  }
  const uint64_t* st = chunks[d.chunk].start + d.sbase;
  span[2 * q] = st[1];
  span[2 * q + 1] = st[d.R - 1] + 1;
}

__device__ __forceinline__ float warp_sum_f(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ long long warp_max_ll(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long t = __shfl_xor_sync(0xffffffffu, v, o);
    v = t > v ? t : v;
  }
  return v;
}

// one warp per leaf: leaf l of query q receives the ids [base, end), base =
// llo + (l << shift), end = base + 2^shift (the last leaf ends at lhi); its
// ranges are first .. last (local indices: the ranges holding base and end - 1).
// Least squares of the local index on the leaf-relative start (FP32, centred),
// then the largest prediction errors below and above over every id the leaf
// receives, from the lookup's own arithmetic at the two ends of each range's
// part of the leaf (the prediction is monotone in h).
__global__ void batch_leaf_fit_kernel(const QueryDev* __restrict__ qd,
                                      const ChunkDev* __restrict__ chunks,
                                      const uint32_t* __restrict__ leaf_q, uint64_t total,
                                      LeafRec* __restrict__ leaves) {
  const uint64_t g = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (g >= total) return;
  const QueryDev Q = qd[leaf_q[g]];
  const uint64_t l = g - Q.loff;
  const uint64_t* st = chunks[Q.chunk].start + Q.sbase;
  const uint64_t b0 = Q.llo + (l << Q.lwshift);
  uint64_t b1 = l + 1 == Q.nleaves ? Q.lhi : b0 + (1ull << Q.lwshift);
  if (b1 > Q.lhi) b1 = Q.lhi;
  const uint32_t first = slice_bs(st, Q.R, b0), last = slice_bs(st, Q.R, b1 - 1);
  LeafRec lr;
  lr.base = b0;
  lr.first = first;
  lr.last = last;
  const uint32_t n = last - first + 1;
  float sx = 0.f, sy = 0.f;
  for (uint32_t i = first + lane; i <= last; i += 32) {
    const uint64_t v = st[i] > b0 ? st[i] : b0;
    sx += __ull2float_rn(v - b0);
    sy += (float)(i - first);
  }
  const float inv_n = 1.0f / (float)n;
  const float mx = warp_sum_f(sx) * inv_n, my = warp_sum_f(sy) * inv_n;
  float sxx = 0.f, sxy = 0.f;
  for (uint32_t i = first + lane; i <= last; i += 32) {
    const uint64_t v = st[i] > b0 ? st[i] : b0;
    const float dx = __ull2float_rn(v - b0) - mx, dy = (float)(i - first) - my;
    sxx = fmaf(dx, dx, sxx);
    sxy = fmaf(dx, dy, sxy);
  }
  sxx = warp_sum_f(sxx);
  sxy = warp_sum_f(sxy);
  const float slope = (sxx > 0.f && sxy > 0.f) ? sxy / sxx : 0.f;
  lr.a = slope;
  lr.b = my - slope * mx;
  lr.errlo = 0;
  lr.errhi = 0;
  long long ehi = 0, elo = 0;
  for (uint32_t i = first + lane; i <= last; i += 32) {
    const uint64_t lo_h = st[i] > b0 ? st[i] : b0;
    const uint64_t hi_h = (st[i + 1] < b1 ? st[i + 1] : b1) - 1;
    const long long plo = (long long)leaf_predict(lr, lo_h);
    const long long phi = (long long)leaf_predict(lr, hi_h);
    const long long up = (long long)i - plo, dn = phi - (long long)i;
    ehi = up > ehi ? up : ehi;
    elo = dn > elo ? dn : elo;
  }
  ehi = warp_max_ll(ehi);
  elo = warp_max_ll(elo);
  const long long CAP = 1ll << 30;
  lr.errhi = (int32_t)(ehi > CAP ? CAP : ehi);
  lr.errlo = (int32_t)(elo > CAP ? CAP : elo);
  if (lane == 0) leaves[g] = lr;
}

}  // namespace
}  // namespace sdb

struct sdb_batch {
  int device = 0;
  uint32_t NP = 0;
  sdb::BatchCore core;
  std::vector<sdb::CoverSet> cs;  // one per chunk of queries
  uint64_t n_ranges = 0, n_cells = 0, max_ranges = 0;
  cudaGraphExec_t graph = nullptr;
  void* g_count = nullptr;
  void* g_sum = nullptr;
};

namespace sdb {
namespace {

template <int G, bool SUM>
sdb_status launch_batch_t(const BatchArgs& A, uint32_t tile, uint32_t lo, uint32_t hi,
                          cudaStream_t s) {
  auto kern = batch_kernel<G, SUM>;
  const uint32_t units = (uint32_t)(((uint64_t)tile + 32 * G - 1) / (32 * G));
  int per_sm = 0;
  SDB_TRY_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, THREADS, 0));
  uint64_t blocks = (uint64_t)num_sms() * (per_sm > 0 ? per_sm : 1);
  const uint64_t need = ((uint64_t)(hi - lo) * units + THREADS / 32 - 1) / (THREADS / 32);
  if (blocks > need) blocks = need;
  if (blocks == 0) return SDB_OK;
  kern<<<(unsigned)blocks, THREADS, 0, s>>>(A, lo, hi, units);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  return SDB_OK;
}

// Points of a lane per unit: the tuning's points per thread, doubled (a unit's two end
// lookups are shared by twice the points), and fewer while the batch's points are not
// enough units for 8 warps per SM (units of 256, 128 and 64 points, one view of 49,000: 21,
// 17 and 15 us; 64 views of 12M: 138, 140 and 214).
sdb_status launch_batch(const BatchArgs& A, uint32_t tile, uint32_t ppt, uint64_t points, bool sum,
                        uint32_t lo, uint32_t hi, cudaStream_t s) {
  uint32_t g = 2 * ppt;
  while (g > 2 && points < (uint64_t)32 * g * 8 * num_sms()) g /= 2;
  if (g == 2) return sum ? launch_batch_t<2, true>(A, tile, lo, hi, s)
                         : launch_batch_t<2, false>(A, tile, lo, hi, s);
  if (g == 4) return sum ? launch_batch_t<4, true>(A, tile, lo, hi, s)
                         : launch_batch_t<4, false>(A, tile, lo, hi, s);
  return sum ? launch_batch_t<8, true>(A, tile, lo, hi, s)
             : launch_batch_t<8, false>(A, tile, lo, hi, s);
}

bool valid_device(int dev) {
  int cur = -1;
  return cudaGetDevice(&cur) == cudaSuccess && cur == dev;
}

sdb_status status_of(cudaError_t e, const char* what) {
  return e == cudaSuccess ? SDB_OK : cuda_status(e, what, __FILE__, __LINE__);
}

}  // namespace

void BatchCore::release(cudaStream_t s) {
  dfree(leaves, s);
  dfree(fallbacks, s);
  leaves = nullptr;
  fallbacks = nullptr;
  dfree(dq, s);
  dfree(dchunks, s);
  dfree(cand, s);
  dfree(ncand, s);
  dfree(tiles, s);
  dq = nullptr;
  dchunks = nullptr;
  cand = nullptr;
  ncand = nullptr;
  tiles = nullptr;
}

sdb_status batch_query_dev(uint32_t B, const sdb_query& Qu, uint64_t out_off, BatchQueryDev* d,
                           uint32_t* F_out) {
  uint32_t k = 0, F = 0;
  SDB_TRY(sdb_finest_level(B, Qu.eps, &k, &F));
  const uint32_t G = 1u << B;
  if (!(Qu.x0 < Qu.x1 && Qu.y0 < Qu.y1 && Qu.x1 <= G && Qu.y1 <= G)) {
    set_error("viewport must be non-empty and inside the grid");
    return SDB_EINVAL;
  }
  memset(d, 0, sizeof(*d));
  d->k = k;
  d->x0 = Qu.x0;
  d->y0 = Qu.y0;
  d->x1 = Qu.x1;
  d->y1 = Qu.y1;
  d->out_off = (uint32_t)out_off;
  *F_out = F;
  return SDB_OK;
}

// The kernel's grid takes every tile for as many units as the largest may have, and most
// ranges of a view are short, so the kernel's tiles are pieces of at most PIECE points
// whatever size is set: one unit of the longest kind.  512 views over 50M points take
// 245 us with 4096-point tiles, 186 with pieces of 1024, 177 with 512, 167 with 256; 4,096
// views over 200M 5.43, 5.16, 4.80 and 4.88 ms.  A tile of "everything" would be 2^26 units
// for each of a batch's thousands of ranges, seconds of them.
constexpr uint32_t PIECE = 256;
sdb_status batch_core_tiles(BatchCore* c, uint32_t T, cudaStream_t s) {
  Scratch sc(s);
  uint64_t *nt, *toff, *dtot;
  SDB_TRY(sc.get(&nt, c->Q));
  SDB_TRY(sc.get(&toff, (size_t)c->Q + 3));
  SDB_TRY(sc.get(&dtot, 3));
  std::vector<uint64_t> off((size_t)c->Q + 3, 0);  // offsets, total, tiles asked for, longest
  uint32_t piece = std::min(T, PIECE);
  for (;;) {
    SDB_TRY_CUDA(cudaMemsetAsync(dtot, 0, 24, s));
    tile_count_kernel<<<grid_for(c->Q, 128), 128, 0, s>>>(
        c->cand, c->ncand, c->Q, piece, T, nt, reinterpret_cast<unsigned long long*>(dtot + 1));
    note_launch();
    SDB_TRY_CUDA(cudaGetLastError());
    SDB_TRY(exclusive_scan<uint64_t>(nt, toff, c->Q, dtot, s));
    SDB_TRY_CUDA(cudaMemcpyAsync(toff + c->Q, dtot, 24, cudaMemcpyDeviceToDevice, s));
    SDB_TRY_CUDA(cudaMemcpyAsync(off.data(), toff, off.size() * 8, cudaMemcpyDeviceToHost, s));
    SDB_TRY_CUDA(cudaStreamSynchronize(s));
    if (off[c->Q] < 0xffffffffull || piece == T) break;
    piece = piece > T / 2 ? T : 2 * piece;  // larger pieces when there are too many
  }
  const uint64_t total = off[c->Q];
  if (total >= 0xffffffffull) {
    set_error("batch: %llu tiles exceed the 32-bit range", (unsigned long long)total);
    return SDB_EINVAL;
  }
  if (c->tiles) dfree(c->tiles, s);
  c->tiles = nullptr;
  SDB_TRY(dalloc_n(&c->tiles, total, s));
  tile_fill_kernel<<<c->Q, 128, 0, s>>>(c->cand, c->ncand, piece, toff, c->tiles);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  SDB_TRY_CUDA(cudaStreamSynchronize(s));
  c->ntiles = off[(size_t)c->Q + 1];
  c->piece = (uint32_t)std::min<uint64_t>(piece, std::max<uint64_t>(off[(size_t)c->Q + 2], 1));
  off.resize((size_t)c->Q + 1);
  c->qtile = std::move(off);
  c->tile = T;
  return SDB_OK;
}

sdb_status batch_core_prepare(BatchCore* c, cudaStream_t s) {
  const uint32_t Q = c->Q;
  SDB_TRY(dalloc_n(&c->dq, Q, s));
  SDB_TRY(dalloc_n(&c->dchunks, c->hchunks.size(), s));
  SDB_TRY(dalloc_n(&c->cand, (size_t)Q * MAXC * 2, s));
  SDB_TRY(dalloc_n(&c->ncand, Q, s));
  SDB_TRY_CUDA(cudaMemcpyAsync(c->dq, c->hq.data(), Q * sizeof(BatchQueryDev),
                               cudaMemcpyHostToDevice, s));
  if (!c->hchunks.empty())
    SDB_TRY_CUDA(cudaMemcpyAsync(c->dchunks, c->hchunks.data(),
                                 c->hchunks.size() * sizeof(BatchChunkDev), cudaMemcpyHostToDevice,
                                 s));
  candidates_kernel<<<Q, CAND_THREADS, 0, s>>>(c->dq, Q, c->pts->key, c->pts->n, c->pts->B, c->cand,
                                               c->ncand);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  SDB_TRY(batch_core_tiles(c, c->tile, s));
  // candidate points (for reporting)
  std::vector<uint32_t> hc((size_t)Q * MAXC * 2), hn(Q);
  SDB_TRY_CUDA(cudaMemcpyAsync(hc.data(), c->cand, hc.size() * 4, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaMemcpyAsync(hn.data(), c->ncand, hn.size() * 4, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaStreamSynchronize(s));
  c->candidates = 0;
  for (uint32_t q = 0; q < Q; ++q)
    for (uint32_t i = 0; i < hn[q]; ++i)
      c->candidates += hc[(size_t)q * MAXC * 2 + 2 * i + 1] - hc[(size_t)q * MAXC * 2 + 2 * i];
  return SDB_OK;
}

sdb_status batch_core_index(BatchCore* c, uint32_t min_ranges, uint32_t ranges_per_leaf,
                            cudaStream_t s) {
  const uint32_t Q = c->Q;
  dfree(c->leaves, s);
  c->leaves = nullptr;
  c->nleaves = 0;
  c->indexed = 0;
  c->learned = min_ranges > 0;
  for (auto& d : c->hq) d.nleaves = d.loff = d.lwshift = 0, d.llo = d.lhi = 0;
  if (c->learned) {
    if (ranges_per_leaf == 0) ranges_per_leaf = 1;
    Scratch sc(s);
    uint64_t* dspan;
    SDB_TRY(sc.get(&dspan, (size_t)Q * 2));
    slice_span_kernel<<<grid_for(Q, 128), 128, 0, s>>>(c->dq, Q, c->dchunks, min_ranges, dspan);
    note_launch();
    SDB_TRY_CUDA(cudaGetLastError());
    std::vector<uint64_t> span((size_t)Q * 2);
    SDB_TRY_CUDA(cudaMemcpyAsync(span.data(), dspan, span.size() * 8, cudaMemcpyDeviceToHost, s));
    SDB_TRY_CUDA(cudaStreamSynchronize(s));
    std::vector<uint32_t> leaf_q;
    uint64_t total = 0;
    for (uint32_t q = 0; q < Q; ++q) {
      BatchQueryDev& d = c->hq[q];
      const uint64_t lo = span[2 * q], hi = span[2 * q + 1];
      if (hi <= lo) continue;  // too few ranges: binary search
      // leaves for about ranges_per_leaf ranges each, a power of two in 16 .. 2^16
      uint64_t want = 16;
      while (want < 65536 && want * ranges_per_leaf < d.R) want *= 2;
      const uint64_t sp = hi - lo;
      uint32_t ws = 0;
      while (((sp + (1ull << ws) - 1) >> ws) > want) ++ws;
      const uint64_t L = (sp + (1ull << ws) - 1) >> ws;
      d.nleaves = (uint32_t)L;
      d.lwshift = ws;
      d.loff = (uint32_t)total;
      d.llo = lo;
      d.lhi = hi;
      total += L;
      if (total >= 0xffffffffull) {
        set_error("batch learned index: %llu leaves exceed the 32-bit range",
                  (unsigned long long)total);
        return SDB_EINVAL;
      }
      leaf_q.insert(leaf_q.end(), (size_t)L, q);
      ++c->indexed;
    }
    if (total) {
      uint32_t* dlq;
      SDB_TRY(sc.get(&dlq, total));
      SDB_TRY(dalloc_n(&c->leaves, total, s));
      if (reinterpret_cast<uintptr_t>(c->leaves) & 31u) {  // leaves are read 32 bytes at once
        set_error("batch learned index: leaf records not 32-byte aligned");
        return SDB_ECUDA;
      }
      SDB_TRY_CUDA(cudaMemcpyAsync(dlq, leaf_q.data(), total * 4, cudaMemcpyHostToDevice, s));
      SDB_TRY_CUDA(cudaMemcpyAsync(c->dq, c->hq.data(), Q * sizeof(BatchQueryDev),
                                   cudaMemcpyHostToDevice, s));
      batch_leaf_fit_kernel<<<grid_for(total * 32, 256), 256, 0, s>>>(c->dq, c->dchunks, dlq,
                                                                      total, c->leaves);
      note_launch();
      SDB_TRY_CUDA(cudaGetLastError());
      SDB_TRY_CUDA(cudaStreamSynchronize(s));
    }
    c->nleaves = total;
    if (!c->fallbacks) {
      SDB_TRY(dalloc_n(&c->fallbacks, 1, s));
      SDB_TRY_CUDA(cudaMemsetAsync(c->fallbacks, 0, sizeof(unsigned long long), s));
    }
  }
  SDB_TRY_CUDA(cudaMemcpyAsync(c->dq, c->hq.data(), Q * sizeof(BatchQueryDev),
                               cudaMemcpyHostToDevice, s));
  SDB_TRY_CUDA(cudaStreamSynchronize(s));
  return SDB_OK;
}

sdb_status batch_core_run(BatchCore* c, int mode, uint64_t* count, int64_t* sum, cudaStream_t s) {
  BatchArgs A;
  A.leaves = c->leaves;
  A.fallbacks = c->fallbacks;
  if (c->fallbacks)
    SDB_TRY_CUDA(cudaMemsetAsync(c->fallbacks, 0, sizeof(unsigned long long), s));
  A.key = c->pts->key;
  A.x = c->pts->x;
  A.y = c->pts->y;
  A.attr = c->pts->attr;
  A.q = c->dq;
  A.tiles = c->tiles;
  A.chunks = c->dchunks;
  A.count = reinterpret_cast<unsigned long long*>(count);
  A.sum = reinterpret_cast<unsigned long long*>(sum);
  if (c->out_len) {
    SDB_TRY_CUDA(cudaMemsetAsync(count, 0, c->out_len * 8, s));
    if (sum) SDB_TRY_CUDA(cudaMemsetAsync(sum, 0, c->out_len * 8, s));
  }
  if (mode == SDB_BATCH_PER_QUERY) {
    for (uint32_t q = 0; q < c->Q; ++q)
      if (c->qtile[q + 1] > c->qtile[q])
        SDB_TRY(launch_batch(A, c->piece, c->ppt,
                             std::min(c->candidates, (c->qtile[q + 1] - c->qtile[q]) * c->piece),
                             sum != nullptr, (uint32_t)c->qtile[q], (uint32_t)c->qtile[q + 1], s));
    return SDB_OK;
  }
  return launch_batch(A, c->piece, c->ppt, c->candidates, sum != nullptr, 0,
                      (uint32_t)c->qtile[c->Q], s);
}

// Coverings of queries [q0, q0 + nq) of a pair list, built in chunks that are
// halved and retried when they overflow the builder's 32-bit ranges or memory.
// Appends CoverSets to *sets and fills sbase/R/chunk of hq.
// Only the polygons that some pair of a chunk names go to the builder (and the
// device): a batch of views meets a few hundred of the 40,000 tracts, and uploading
// all of their 900k vertices per batch took as long as building the coverings.
sdb_status build_query_coverings(const PolySet& polys, uint32_t B,
                                 const std::vector<CoverQuery>& cq,
                                 const std::vector<uint32_t>& pp, const std::vector<uint32_t>& pq,
                                 const std::vector<uint32_t>& ps, std::vector<BatchQueryDev>& hq,
                                 std::vector<CoverSet>* sets, uint32_t chunk_base,
                                 cudaStream_t s, uint64_t* n_ranges, uint64_t* n_cells,
                                 uint64_t* max_ranges) {
  const uint32_t Q = (uint32_t)cq.size();
  std::vector<uint64_t> pfirst((size_t)Q + 1, 0);  // pairs are in query order
  for (uint64_t i = 0, q = 0; q <= Q; ++q) {
    while (i < pq.size() && pq[i] < q) ++i;
    pfirst[q] = i;
  }
  uint32_t chunk_q = 512;
  std::vector<uint32_t> pq_local, pp_local, cx, cy, local(polys.P, NONE);
  for (uint32_t q0 = 0; q0 < Q;) {
    // queries of a chunk share 64-bit keys: query bits above 2 * (finest level)
    uint32_t nq = std::min(chunk_q, Q - q0);
    for (;;) {
      uint32_t Fm = 0;
      for (uint32_t q = q0; q < q0 + nq; ++q) Fm = std::max(Fm, cq[q].F);
      const uint32_t room = 64 - 2 * Fm;  // F <= 30
      if (nq == 1 || room >= 32 || nq <= (1u << room)) break;
      nq = 1u << room;
    }
    const uint64_t pa = pfirst[q0], pb = pfirst[q0 + nq];
    pq_local.assign(pq.begin() + pa, pq.begin() + pb);
    for (auto& v : pq_local) v -= q0;
    PolyEdges pe;
    pe.edge_off.push_back(0);
    pp_local.resize(pb - pa);
    cx.clear();
    cy.clear();
    for (uint64_t i = pa; i < pb; ++i) {
      const uint32_t j = pp[i], v0 = polys.off[j], v1 = polys.off[j + 1];
      if (local[j] == NONE) {
        local[j] = pe.P++;
        const uint32_t at = (uint32_t)cx.size();
        cx.insert(cx.end(), polys.x + v0, polys.x + v1);
        cy.insert(cy.end(), polys.y + v0, polys.y + v1);
        for (uint32_t v = v0; v < v1; ++v)
          pe.next.push_back(at + (polys.next ? polys.next[v] - v0 : v + 1 < v1 ? v + 1 - v0 : 0));
        pe.edge_off.push_back((uint32_t)cx.size());
      }
      pp_local[i - pa] = local[j];
    }
    for (uint64_t i = pa; i < pb; ++i) local[pp[i]] = NONE;
    pe.V = (uint32_t)cx.size();
    pe.x = cx.data();
    pe.y = cy.data();
    CoverSpec spec;
    spec.B = B;
    spec.Q = nq;
    spec.q = cq.data() + q0;
    spec.NP = (uint32_t)(pb - pa);
    spec.pair_poly = pp_local.data();
    spec.pair_query = pq_local.data();
    spec.pair_slot = ps.data() + pa;
    CoverSet set;
    sdb_status st = build_coverings(pe, spec, s, &set);
    if (st == SDB_ENOMEM && nq > 1) {
      set.release(s);
      cudaStreamSynchronize(s);
      cudaGetLastError();
      chunk_q = nq / 2;
      continue;
    }
    if (st != SDB_OK) {
      set.release(s);
      return st;
    }
    for (uint32_t q = 0; q < nq; ++q) {
      BatchQueryDev& d = hq[q0 + q];
      d.sbase = set.qoff[q];
      d.R = (uint32_t)(set.qoff[q + 1] - set.qoff[q] - 1);
      d.chunk = chunk_base + (uint32_t)sets->size();
      *max_ranges = std::max<uint64_t>(*max_ranges, d.R);
    }
    *n_ranges += set.E - nq;
    *n_cells += set.ncells;
    sets->push_back(set);
    q0 += nq;
  }
  return SDB_OK;
}

// (query, polygon) pairs whose polygon's cells can hold viewport points: the
// polygon's bounding box grown by one finest cell meets the viewport
void viewport_pairs(const std::vector<uint32_t>& bb, uint32_t q, const sdb_query& Qu, uint32_t k,
                    const uint32_t* ids, std::vector<uint32_t>& pp, std::vector<uint32_t>& pq,
                    std::vector<uint32_t>& ps) {
  const int64_t g = (int64_t)1 << k;
  for (uint32_t t = 0; t < Qu.poly_cnt; ++t) {
    const uint32_t j = ids[t];
    if ((int64_t)bb[4 * j] - g < (int64_t)Qu.x1 && (int64_t)bb[4 * j + 2] + g >= Qu.x0 &&
        (int64_t)bb[4 * j + 1] - g < (int64_t)Qu.y1 && (int64_t)bb[4 * j + 3] + g >= Qu.y0) {
      pp.push_back(j);
      pq.push_back(q);
      ps.push_back(t);
    }
  }
}

sdb_status polygon_bboxes(const sdb_polygons* polys, uint32_t B, std::vector<uint32_t>* bb) {
  const uint32_t P = polys->n_polygons, G = 1u << B;
  if (P == 0 || P >= (1u << 26) || polys->ring_off[0] != 0) {
    set_error("bad polygon set");
    return SDB_EINVAL;
  }
  bb->assign(4ull * P, 0);
  for (uint32_t j = 0; j < P; ++j) {
    if (polys->ring_off[j + 1] < polys->ring_off[j] + 3) {
      set_error("polygon %u has fewer than 3 vertices", j);
      return SDB_EINVAL;
    }
    uint32_t mnx = ~0u, mny = ~0u, mxx = 0, mxy = 0;
    const uint32_t v0 = polys->ring_off[j], v1 = polys->ring_off[j + 1];
    for (uint32_t v = v0; v < v1; ++v) {
      mnx = std::min(mnx, polys->x[v]);
      mxx = std::max(mxx, polys->x[v]);
      mny = std::min(mny, polys->y[v]);
      mxy = std::max(mxy, polys->y[v]);
    }
    if (mxx >= G || mxy >= G) {
      uint32_t v = v0;
      while (polys->x[v] < G && polys->y[v] < G) ++v;
      set_error("vertex %u outside the grid", v);
      return SDB_EINVAL;
    }
    (*bb)[4 * j] = mnx;
    (*bb)[4 * j + 1] = mny;
    (*bb)[4 * j + 2] = mxx;
    (*bb)[4 * j + 3] = mxy;
  }
  return SDB_OK;
}

}  // namespace sdb

using namespace sdb;

extern "C" {

sdb_status sdb_points_create(const uint32_t* d_x, const uint32_t* d_y, const int32_t* d_attr,
                             uint64_t n, uint32_t grid_bits, void* cuda_stream, sdb_points** out) {
  if (!out) {
    set_error("out is NULL");
    return SDB_EINVAL;
  }
  *out = nullptr;
  if (grid_bits < 1 || grid_bits > 30) {
    set_error("grid_bits %u outside 1..30", grid_bits);
    return SDB_EINVAL;
  }
  if (n == 0 || n >= 0xffffffffull || !d_x || !d_y) {
    set_error("need 1 <= n < 2^32 points with coordinates");
    return SDB_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)cuda_stream;
  sdb_points* p = new (std::nothrow) sdb_points();
  if (!p) {
    set_error("host allocation failed");
    return SDB_ENOMEM;
  }
  cudaGetDevice(&p->device);
  p->B = grid_bits;
  p->n = n;
  sdb_status st = SDB_OK;
  {
    Scratch sc(s);
    uint64_t *ktmp = nullptr, *ks = nullptr;
    uint32_t *vtmp = nullptr, *vs = nullptr;
    unsigned int* bad = nullptr;
    uint32_t nsteps, st0;
    hilbert3_params(grid_bits, &nsteps, &st0);
    st = dalloc_n(&p->key, n, s);
    if (st == SDB_OK) st = dalloc_n(&p->attr, n, s);
    if (st == SDB_OK) st = dalloc_n(&ktmp, n, s);
    if (st == SDB_OK && d_attr) st = dalloc_n(&vtmp, n, s);
    if (st == SDB_OK) st = sc.get(&bad, 1);
    if (st == SDB_OK) st = status_of(cudaMemsetAsync(bad, 0, 4, s), "memset");
    if (st == SDB_OK) {
      const int vec = (((uintptr_t)d_x | (uintptr_t)d_y) & 15u) == 0;
      const unsigned grid = std::min<unsigned>(num_sms() * 8, grid_for((n + 3) / 4, 256));
      point_keys_kernel<<<grid, 256, 0, s>>>(d_x, d_y, n, grid_bits, nsteps, st0, vec, p->key,
                                             bad);
      note_launch();
      st = status_of(cudaGetLastError(), "point keys");
    }
    // keys with their attributes; the buffer that ends up sorted is kept
    if (st == SDB_OK && d_attr) {
      uint32_t* va = reinterpret_cast<uint32_t*>(p->attr);
      st = radix_sort_pairs(p->key, va, ktmp, vtmp, n, 2 * grid_bits, s, &ks, &vs,
                            reinterpret_cast<const uint32_t*>(d_attr));
      if (st == SDB_OK && vs != va) {
        p->attr = reinterpret_cast<int32_t*>(vs);
        vtmp = va;
      }
    } else if (st == SDB_OK) {
      st = status_of(cudaMemsetAsync(p->attr, 0, n * 4, s), "memset");
      if (st == SDB_OK) st = radix_sort_keys(p->key, ktmp, n, 2 * grid_bits, s, &ks);
    }
    if (st == SDB_OK && ks != p->key) std::swap(p->key, ktmp);
    dfree(ktmp, s);
    dfree(vtmp, s);
    if (st == SDB_OK) st = dalloc_n(&p->x, n, s);
    if (st == SDB_OK) st = dalloc_n(&p->y, n, s);
    if (st == SDB_OK) {
      const unsigned grid = std::min<unsigned>(num_sms() * 8, grid_for((n + 3) / 4, 256));
      point_coords_kernel<<<grid, 256, 0, s>>>(p->key, n, nsteps, st0, p->x, p->y);
      note_launch();
      st = status_of(cudaGetLastError(), "point coordinates");
    }
    if (st == SDB_OK) {
      unsigned int hb = 0;
      st = status_of(cudaMemcpyAsync(&hb, bad, 4, cudaMemcpyDeviceToHost, s), "flag copy");
      if (st == SDB_OK) st = status_of(cudaStreamSynchronize(s), "points create");
      if (st == SDB_OK && hb) {
        set_error("a point lies outside the grid [0, 2^%u)", grid_bits);
        st = SDB_EINVAL;
      }
    }
  }
  if (st != SDB_OK) {
    sdb_points_free(p);
    return st;
  }
  *out = p;
  return SDB_OK;
}

void sdb_points_free(sdb_points* p) {
  if (!p) return;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(p->device);
  cudaDeviceSynchronize();
  sdb::release_point_index(p, 0);
  void* ps[] = {p->key, p->x, p->y, p->attr};
  for (void* q : ps)
    if (q) cudaFreeAsync(q, 0);
  cudaStreamSynchronize(0);
  cudaSetDevice(prev);
  delete p;
}

sdb_status sdb_batch_create(const sdb_points* pts, const sdb_polygons* polys,
                            const sdb_query* queries, uint32_t n_queries,
                            const uint32_t* subset_ids, uint64_t n_subset_ids, void* cuda_stream,
                            sdb_batch** out) {
  if (!out || !pts || !polys || !queries || n_queries == 0 || !polys->ring_off || !polys->x ||
      !polys->y) {
    set_error("points, polygons, queries and out are required");
    return SDB_EINVAL;
  }
  *out = nullptr;
  if (!valid_device(pts->device)) {
    set_error("points live on another device");
    return SDB_EINVAL;
  }
  const uint32_t B = pts->B, P = polys->n_polygons;
  std::vector<uint32_t> bb;
  SDB_TRY(polygon_bboxes(polys, B, &bb));
  std::vector<CoverQuery> cq(n_queries);
  std::vector<BatchQueryDev> hq(n_queries);
  std::vector<uint32_t> pp, pq, ps;
  uint64_t out_off = 0;
  for (uint32_t q = 0; q < n_queries; ++q) {
    const sdb_query& Qu = queries[q];
    uint32_t F = 0;
    sdb_status st = batch_query_dev(B, Qu, out_off, &hq[q], &F);
    if (st != SDB_OK) {
      set_error("query %u: %s", q, std::string(sdb_last_error()).c_str());
      return st;
    }
    if ((uint64_t)Qu.poly_off + Qu.poly_cnt > n_subset_ids || (Qu.poly_cnt && !subset_ids)) {
      set_error("query %u: polygon subset outside the id array", q);
      return SDB_EINVAL;
    }
    for (uint32_t t = 0; t < Qu.poly_cnt; ++t)
      if (subset_ids[Qu.poly_off + t] >= P) {
        set_error("query %u: polygon id %u out of range", q, subset_ids[Qu.poly_off + t]);
        return SDB_EINVAL;
      }
    if (out_off + Qu.poly_cnt >= 0xffffffffull) {
      set_error("batch output exceeds 2^32 entries");
      return SDB_EINVAL;
    }
    cq[q] = CoverQuery{F, Qu.x0, Qu.y0, Qu.x1, Qu.y1};
    viewport_pairs(bb, q, Qu, hq[q].k, subset_ids ? subset_ids + Qu.poly_off : nullptr, pp, pq,
                   ps);
    out_off += Qu.poly_cnt;
  }
  cudaStream_t s = (cudaStream_t)cuda_stream;
  sdb_batch* b = new (std::nothrow) sdb_batch();
  if (!b) {
    set_error("host allocation failed");
    return SDB_ENOMEM;
  }
  b->device = pts->device;
  b->NP = (uint32_t)pp.size();
  b->core.pts = pts;
  b->core.Q = n_queries;
  b->core.out_len = out_off;
  sdb_status st = build_query_coverings(PolySet{P, polys->ring_off, polys->x, polys->y, nullptr}, B, cq, pp, pq, ps, hq, &b->cs, 0, s,
                                        &b->n_ranges, &b->n_cells, &b->max_ranges);
  if (st == SDB_OK) {
    b->core.hq = hq;
    for (auto& c : b->cs)
      b->core.hchunks.push_back(BatchChunkDev{c.start, c.pay, c.list_off, c.list_ids});
    st = batch_core_prepare(&b->core, s);
  }
  if (st != SDB_OK) {
    std::string msg = sdb_last_error();
    sdb_batch_free(b);
    set_error("%s", msg.c_str());
    return st;
  }
  *out = b;
  return SDB_OK;
}

sdb_status sdb_batch_get_info(const sdb_batch* b, sdb_batch_info* info) {
  if (!b || !info) {
    set_error("batch or info is NULL");
    return SDB_EINVAL;
  }
  memset(info, 0, sizeof(*info));
  info->n_queries = b->core.Q;
  info->n_pairs = b->NP;
  info->out_len = b->core.out_len;
  info->n_ranges = b->n_ranges;
  info->max_ranges = b->max_ranges;
  info->n_cells = b->n_cells;
  info->candidates = b->core.candidates;
  info->n_tiles = b->core.ntiles;
  info->tile = b->core.tile;
  info->points_per_thread = b->core.ppt;
  info->lookup = b->core.learned ? SDB_LOOKUP_LEARNED : SDB_LOOKUP_BINARY;
  info->indexed_queries = b->core.indexed;
  info->n_leaves = b->core.nleaves;
  return SDB_OK;
}

sdb_status sdb_batch_set_lookup(sdb_batch* b, int lookup, void* cuda_stream) {
  if (!b || (lookup != SDB_LOOKUP_BINARY && lookup != SDB_LOOKUP_LEARNED)) {
    set_error("batch NULL, or a lookup other than binary search and the learned index");
    return SDB_EINVAL;
  }
  if (!valid_device(b->device)) {
    set_error("batch lives on another device");
    return SDB_EINVAL;
  }
  if (b->graph) {  // the captured launch refers to the old lookup structures
    cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
  }
  return batch_core_index(&b->core, lookup == SDB_LOOKUP_LEARNED ? SDB_BATCH_LEARNED_MIN_RANGES : 0,
                          SDB_BATCH_RANGES_PER_LEAF, (cudaStream_t)cuda_stream);
}

sdb_status sdb_batch_fallbacks(const sdb_batch* b, void* cuda_stream, uint64_t* out) {
  if (!b || !out) {
    set_error("batch or output is NULL");
    return SDB_EINVAL;
  }
  *out = 0;
  if (!b->core.fallbacks) return SDB_OK;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  SDB_TRY_CUDA(cudaMemcpyAsync(out, b->core.fallbacks, 8, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaStreamSynchronize(s));
  return SDB_OK;
}

sdb_status sdb_batch_run(sdb_batch* b, int mode, uint64_t* d_count, int64_t* d_sum,
                         void* cuda_stream) {
  if (!b || !d_count) {
    set_error("batch or d_count is NULL");
    return SDB_EINVAL;
  }
  if (!valid_device(b->device)) {
    set_error("batch lives on another device");
    return SDB_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)cuda_stream;
  if (mode == SDB_BATCH_PERSISTENT || mode == SDB_BATCH_PER_QUERY)
    return batch_core_run(&b->core, mode, d_count, d_sum, s);
  if (mode == SDB_BATCH_GRAPH) {
    if (s == nullptr) {
      set_error("graph mode needs a created stream (the legacy stream cannot be captured)");
      return SDB_EINVAL;
    }
    if (!b->graph || b->g_count != d_count || b->g_sum != d_sum) {
      if (b->graph) {
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
      }
      cudaGraph_t g = nullptr;
      SDB_TRY_CUDA(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
      sdb_status st = batch_core_run(&b->core, SDB_BATCH_PERSISTENT, d_count, d_sum, s);
      cudaError_t e = cudaStreamEndCapture(s, &g);
      if (st != SDB_OK) {
        if (g) cudaGraphDestroy(g);
        return st;
      }
      if (e != cudaSuccess) return cuda_status(e, "cudaStreamEndCapture", __FILE__, __LINE__);
      e = cudaGraphInstantiate(&b->graph, g, 0);
      cudaGraphDestroy(g);
      if (e != cudaSuccess) {
        b->graph = nullptr;
        return cuda_status(e, "cudaGraphInstantiate", __FILE__, __LINE__);
      }
      b->g_count = d_count;
      b->g_sum = d_sum;
    }
    SDB_TRY_CUDA(cudaGraphLaunch(b->graph, s));
    return SDB_OK;
  }
  set_error("unknown batch mode %d", mode);
  return SDB_EINVAL;
}

static sdb_status set_tiles(sdb_batch* b, uint32_t T, cudaStream_t s) {
  SDB_TRY(batch_core_tiles(&b->core, T, s));
  if (b->graph) {  // the captured launch refers to the old work list
    cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
  }
  return SDB_OK;
}

sdb_status sdb_batch_autotune(sdb_batch* b, void* cuda_stream, uint32_t* tile_out,
                              uint32_t* ppt_out) {
  if (!b) {
    set_error("batch is NULL");
    return SDB_EINVAL;
  }
  if (!valid_device(b->device)) {
    set_error("batch lives on another device");
    return SDB_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)cuda_stream;
  Scratch sc(s);
  uint64_t* cnt;
  int64_t* sm;
  SDB_TRY(sc.get(&cnt, b->core.out_len));
  SDB_TRY(sc.get(&sm, b->core.out_len));
  cudaEvent_t e0, e1;
  SDB_TRY_CUDA(cudaEventCreate(&e0));
  SDB_TRY_CUDA(cudaEventCreate(&e1));
  const uint32_t tiles[] = {1024, 4096, 16384};
  const uint32_t ppts[] = {1, 2, 4};
  float best = 1e30f;
  uint32_t bt = b->core.tile, bp = b->core.ppt;
  sdb_status st = SDB_OK;
  for (uint32_t T : tiles) {
    if ((st = set_tiles(b, T, s)) != SDB_OK) break;
    for (uint32_t G : ppts) {
      b->core.ppt = G;
      float ms = 0;
      for (int rep = 0; rep < 2 && st == SDB_OK; ++rep) {  // the first run warms up
        cudaEventRecord(e0, s);
        st = batch_core_run(&b->core, SDB_BATCH_PERSISTENT, cnt, sm, s);
        cudaEventRecord(e1, s);
        if (cudaEventSynchronize(e1) != cudaSuccess) st = SDB_ECUDA;
        cudaEventElapsedTime(&ms, e0, e1);
      }
      if (st != SDB_OK) break;
      if (ms < best) {
        best = ms;
        bt = T;
        bp = G;
      }
    }
    if (st != SDB_OK) break;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  b->core.ppt = bp;
  if (st == SDB_OK) st = set_tiles(b, bt, s);
  if (st == SDB_OK) {
    if (tile_out) *tile_out = bt;
    if (ppt_out) *ppt_out = bp;
  }
  return st;
}

sdb_status sdb_batch_set_tuning(sdb_batch* b, uint32_t tile, uint32_t points_per_thread,
                                void* cuda_stream) {
  if (!b || tile == 0 || !(points_per_thread == 1 || points_per_thread == 2 ||
                           points_per_thread == 4)) {
    set_error("batch NULL, tile 0, or points per thread not 1, 2 or 4");
    return SDB_EINVAL;
  }
  b->core.ppt = points_per_thread;
  return set_tiles(b, tile, (cudaStream_t)cuda_stream);
}

sdb_status sdb_batch_query_ranges(const sdb_batch* b, uint32_t* h_ranges) {
  if (!b || !h_ranges) {
    set_error("batch or output is NULL");
    return SDB_EINVAL;
  }
  for (uint32_t q = 0; q < b->core.Q; ++q) h_ranges[q] = b->core.hq[q].R;
  return SDB_OK;
}

void sdb_batch_free(sdb_batch* b) {
  if (!b) return;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(b->device);
  cudaDeviceSynchronize();
  if (b->graph) cudaGraphExecDestroy(b->graph);
  for (auto& c : b->cs) c.release(0);
  b->core.release(0);
  cudaStreamSynchronize(0);
  cudaSetDevice(prev);
  delete b;
}

}  // extern "C"
