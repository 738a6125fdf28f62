// Point-indexed aggregation (Sec. 3, "Point Indexing").  The resident points
// are already ordered by their full-resolution Hilbert id (level B); a covering
// range [h, h') at the finest level F holds exactly the points whose ids lie in
// [h << 2k, h' << 2k) (the curve's prefix property), a contiguous slice of the
// sorted array.  COUNT is the slice's length and SUM a difference of prefix
// sums, so one lower-bound lookup per range boundary answers the whole
// covering.  The lookups use binary search or a RadixSpline (the paper's learned
// index: spline points with a bounded interpolation error and a radix table over
// the keys' top bits).
//
//  * prefix[i] = attr[0] + ... + attr[i-1] in key order, int64 (n + 1 entries).
//  * spline: over the distinct keys (each at its first position), the greedy
//    spline corridor: from the last spline point, keep the narrowest cone of
//    slopes that passes within +-E of every point seen; when a point leaves the
//    cone the previous point becomes a spline point.  Slopes are compared exactly
//    (128-bit cross products where FP32 does not settle them).  The array is cut
//    into chunks of CHUNK keys, each scanned by one warp, every chunk starting and
//    ending with a spline point (one pass, in parallel; the bound holds on every
//    segment).
//  * radix table: entry j = first spline point whose key, minus the smallest
//    key, shifted right so that 2^radix_bits prefixes cover the key range, is
//    >= j.  A lookup reads two entries, searches the few spline points between
//    them, interpolates exactly in integers, and searches +-(E + 1) around the
//    estimate; the bracket is verified and plain binary search is the fallback
//    (counted).
#include "sdb_internal.cuh"

namespace sdb {

namespace {

constexpr uint64_t CHUNK = 4096;  // keys per independent stretch of the spline
constexpr uint32_t NONE = 0xffffffffu;

struct SplinePt {
  uint64_t k;
  int64_t p;
};

// slope(a -> b1) < slope(a -> b2), both keys above a's
__device__ __forceinline__ bool slope_less(const SplinePt& a, const SplinePt& b1,
                                           const SplinePt& b2) {
  const __int128 l = (__int128)(b1.p - a.p) * (__int128)(b2.k - a.k);
  const __int128 r = (__int128)(b2.p - a.p) * (__int128)(b1.k - a.k);
  return l < r;
}

constexpr uint32_t FULL = 0xffffffffu;
constexpr int SPLINE_WARPS = 4;             // chunks per block
constexpr uint32_t MASK_WORDS = CHUNK / 32;  // spline-point bits of a chunk

// Does the distinct key at position j leave the cone of its segment (base, then
// the distinct keys in (base, j))?  Exact, the warp's lanes over the segment.
__device__ __noinline__ bool leaves_cone_exact(const uint64_t* __restrict__ key, uint64_t base,
                                               uint64_t j, int64_t E) {
  const SplinePt b{key[base], (int64_t)base}, cp{key[j], (int64_t)j};
  bool out = false;
  for (uint64_t i = base + 1 + (threadIdx.x & 31); i < j; i += 32) {
    const uint64_t k = key[i];
    if (k == key[i - 1]) continue;
    out |= slope_less(b, SplinePt{k, (int64_t)i + E}, cp) ||
           slope_less(b, cp, SplinePt{k, (int64_t)i - E});
  }
  return __any_sync(FULL, out);
}

// The greedy corridor over each chunk's distinct keys, one warp per chunk: 32
// keys a step, the cone's upper and lower slope at every key by warp scans.
// The slopes are FP32 (each within 2^-22 of its value); a key within 2^-20 of an
// edge of the cone is decided by the exact comparison, so the spline is the
// exact greedy one.  The chunk's spline points are left as bits of its mask.
// A thread per chunk, reading 32 KB on its own twice over (to count, then to
// write), took 3.54 ms for 30M keys; this and the write take 0.26 ms.
__global__ __launch_bounds__(SPLINE_WARPS * 32) void spline_mark_kernel(
    const uint64_t* __restrict__ key, uint64_t n, uint64_t nchunks, int64_t E,
    uint32_t* __restrict__ mask, uint64_t* __restrict__ cnt) {
  __shared__ uint32_t s_mask[SPLINE_WARPS][MASK_WORDS];
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint64_t c = (uint64_t)blockIdx.x * SPLINE_WARPS + w;
  if (c >= nchunks) return;  // whole warps leave; no block barrier below
  uint32_t* sm = s_mask[w];
  for (uint32_t i = lane; i < MASK_WORDS; i += 32) sm[i] = 0;
  __syncwarp();
  const uint64_t i0 = c * CHUNK, end = min(n, i0 + CHUNK);
  auto emit = [&](uint64_t p) {
    if (lane == 0) sm[(p - i0) >> 5] |= 1u << ((p - i0) & 31);
  };
  // past a run of equal keys begun in the previous chunk
  uint64_t base = end;
  for (uint64_t j0 = i0; j0 < end && base == end; j0 += 32) {
    const uint64_t j = j0 + lane;
    const uint32_t f = __ballot_sync(FULL, j < end && (j == 0 || key[j] != key[j - 1]));
    if (f) base = j0 + (__ffs(f) - 1);
  }
  if (base < end) {
    constexpr float DELTA = 1.0f / (1 << 20);
    const float inf = __int_as_float(0x7f800000);
    const float Ef = (float)E;
    uint64_t bk = key[base], prev = base;
    float carry_u = inf, carry_l = -inf;  // over the segment's keys before this step
    emit(base);
    for (uint64_t j0 = base + 1; j0 < end;) {
      const uint64_t j = j0 + lane;
      const uint64_t k = j < end ? key[j] : 0ull;
      uint64_t kp = __shfl_up_sync(FULL, k, 1);
      if (lane == 0) kp = key[j0 - 1];
      const bool distinct = j < end && k != kp;
      const float dp = (float)(uint32_t)(j - base);
      const float inv = __frcp_rn(__ull2float_rn(distinct ? k - bk : 1ull));
      float u = distinct ? (dp + Ef) * inv : inf, l = distinct ? (dp - Ef) * inv : -inf;
      const float cs = dp * inv;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const float tu = __shfl_up_sync(FULL, u, o), tl = __shfl_up_sync(FULL, l, o);
        if (lane >= (uint32_t)o) {
          u = fminf(u, tu);
          l = fmaxf(l, tl);
        }
      }
      // the cone as this key finds it: the segment's earlier keys
      float mu = __shfl_up_sync(FULL, u, 1), ml = __shfl_up_sync(FULL, l, 1);
      mu = lane == 0 ? carry_u : fminf(mu, carry_u);
      ml = lane == 0 ? carry_l : fmaxf(ml, carry_l);
      const bool open = distinct && mu < inf;  // a first key after the base is always inside
      const bool out = open && (cs > mu * (1.0f + DELTA) || (ml > 0.f && cs < ml * (1.0f - DELTA)));
      const bool near = open && (cs > mu * (1.0f - DELTA) || (ml > 0.f && cs < ml * (1.0f + DELTA)));
      const uint32_t dmask = __ballot_sync(FULL, distinct);
      const uint32_t omask = __ballot_sync(FULL, out);
      uint32_t cand = __ballot_sync(FULL, near) | omask;
      int leave = -1;
      while (cand) {
        const int t = __ffs(cand) - 1;
        cand &= cand - 1;
        if (((omask >> t) & 1u) || leaves_cone_exact(key, base, j0 + t, E)) {
          leave = t;
          break;
        }
      }
      if (leave < 0) {
        if (dmask) prev = j0 + (31 - __clz(dmask));
        carry_u = fminf(carry_u, __shfl_sync(FULL, u, 31));
        carry_l = fmaxf(carry_l, __shfl_sync(FULL, l, 31));
        j0 += 32;
      } else {  // the key before it ends the segment and starts the next one
        const uint32_t before = dmask & ((1u << leave) - 1u);
        if (before) prev = j0 + (31 - __clz(before));
        emit(prev);
        base = prev;
        bk = key[base];
        carry_u = inf;
        carry_l = -inf;
        j0 += leave;
      }
    }
    if (prev != base) emit(prev);  // the chunk's last distinct key closes it
  }
  __syncwarp();
  uint32_t m = 0;
  for (uint32_t i = lane; i < MASK_WORDS; i += 32) {
    mask[c * MASK_WORDS + i] = sm[i];
    m += __popc(sm[i]);
  }
  m = __reduce_add_sync(FULL, m);
  if (lane == 0) cnt[c] = m;
}

// the marked keys and positions, in order: one warp per chunk, from off[c] on
__global__ __launch_bounds__(SPLINE_WARPS * 32) void spline_write_kernel(
    const uint64_t* __restrict__ key, uint64_t nchunks, const uint32_t* __restrict__ mask,
    const uint64_t* __restrict__ off, uint64_t* __restrict__ sk, uint32_t* __restrict__ sp) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t c = (uint64_t)blockIdx.x * SPLINE_WARPS + (threadIdx.x >> 5);
  if (c >= nchunks) return;
  uint64_t o = off[c];
  for (uint32_t i = 0; i < MASK_WORDS; i += 32) {
    uint32_t b = mask[c * MASK_WORDS + i + lane];
    const uint32_t m = __popc(b);
    uint32_t inc = m;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const uint32_t t = __shfl_up_sync(FULL, inc, s);
      if (lane >= (uint32_t)s) inc += t;
    }
    uint64_t at = o + inc - m;
    for (; b; b &= b - 1) {
      const uint64_t p = c * CHUNK + (uint64_t)(i + lane) * 32 + (__ffs(b) - 1);
      sk[at] = key[p];
      sp[at] = (uint32_t)p;
      ++at;
    }
    o += __shfl_sync(FULL, inc, 31);
  }
}

// first spline point in [lo, hi) with key >= q, hi if none
__device__ __forceinline__ uint32_t spline_lower(const uint64_t* __restrict__ sk, uint32_t lo,
                                                 uint32_t hi, uint64_t q) {
  uint32_t len = hi - lo;
  while (len > 0) {
    const uint32_t half = len >> 1;
    if (__ldg(sk + lo + half) < q) {
      lo += half + 1;
      len -= half + 1;
    } else {
      len = half;
    }
  }
  return lo;
}

// table[j] = first spline point with prefix >= j, j in [0, 2^r]: the prefix of
// key x is (x - kmin) >> shift, which is >= j exactly when x >= kmin + (j << shift).
// A block writes TABLE_TILE entries: it searches the spline for its first and
// last entry only, and the entries between look into the few points between
// those (2^25 entries: a search of the whole spline each took 388 us, this
// 127 us; the 134 MB written are 20).
constexpr uint32_t TABLE_TILE = 16384;
__global__ __launch_bounds__(256) void radix_table_kernel(const uint64_t* __restrict__ sk,
                                                          uint32_t ns, uint64_t kmin,
                                                          uint32_t shift, uint32_t r,
                                                          uint32_t* __restrict__ table) {
  __shared__ uint32_t s_lo, s_hi;
  const uint64_t j0 = (uint64_t)blockIdx.x * TABLE_TILE;
  const uint64_t j1 = min(j0 + TABLE_TILE, ((uint64_t)1 << r) + 1);  // past the block's last entry
  if (threadIdx.x == 0) s_lo = spline_lower(sk, 0, ns, kmin + (j0 << shift));
  if (threadIdx.x == 32) s_hi = spline_lower(sk, 0, ns, kmin + ((j1 - 1) << shift));
  __syncthreads();
  const uint32_t lo = s_lo, hi = s_hi;
  for (uint64_t j = j0 + threadIdx.x; j < j1; j += blockDim.x)
    table[j] = spline_lower(sk, lo, hi, kmin + (j << shift));
}

struct Spline {
  const uint64_t* key;  // the points' sorted keys
  uint64_t n;
  const uint64_t* sk;
  const uint32_t* sp;
  uint64_t ns;
  const uint32_t* table;
  uint64_t kmin, kmax;
  uint32_t shift;
  int64_t E;
  unsigned long long* fallbacks;
};

// first index in [lo, hi) with key >= q, hi if none
__device__ __forceinline__ uint64_t lower_bound_in(const uint64_t* __restrict__ key, uint64_t lo,
                                                   uint64_t hi, uint64_t q) {
  uint64_t len = hi - lo;
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

// the last spline point with key <= q (q within the keys) through the radix table
__device__ __forceinline__ uint32_t spline_segment(const Spline& S, uint64_t q) {
  const uint64_t j = (q - S.kmin) >> S.shift;
  // it lies in [table[j] - 1, table[j + 1])
  uint32_t a = __ldg(S.table + j), b = __ldg(S.table + j + 1);
  a = a > 0 ? a - 1 : 0;
  for (uint32_t len = b - a; len > 1;) {  // sk[a] <= q holds
    const uint32_t half = len >> 1;
    if (__ldg(S.sk + a + half) <= q) a += half;
    len -= half;
  }
  return a;
}

// floor(num * d / den) for num < den: a small quotient (d <= 4096, as between two
// spline points of a chunk) from an FP32 estimate that 128-bit products settle,
// others by the 128-bit division
__device__ __forceinline__ uint64_t interpolate(uint64_t num, uint64_t den, uint64_t d) {
  if (d > 4096) return (uint64_t)((unsigned __int128)num * d / den);
  uint64_t t = (uint64_t)(__ull2float_rn(num) * __frcp_rn(__ull2float_rn(den)) * (float)(uint32_t)d);
  const unsigned __int128 p = (unsigned __int128)num * d;
  if ((unsigned __int128)den * t > p) {
    --t;
  } else if ((unsigned __int128)den * (t + 1) <= p) {
    ++t;
  }
  return t;
}

// lower bound of q (kmin < q <= kmax) given its spline segment a
__device__ __forceinline__ uint64_t spline_position(const Spline& S, uint32_t a, uint64_t q,
                                                    bool counted) {
  uint64_t est = __ldg(S.sp + a);
  if (a + 1 < S.ns) {
    const uint64_t k0 = __ldg(S.sk + a), k1 = __ldg(S.sk + a + 1);
    est += interpolate(q - k0, k1 - k0, (uint64_t)__ldg(S.sp + a + 1) - est);
  }
  const uint64_t lo = est > (uint64_t)S.E + 1 ? est - (uint64_t)S.E - 1 : 0;
  const uint64_t hi = min(S.n, est + (uint64_t)S.E + 2);
  const uint64_t pos = lower_bound_in(S.key, lo, hi, q);
  const bool ok = (pos == 0 || __ldg(S.key + pos - 1) < q) && (pos == S.n || __ldg(S.key + pos) >= q);
  if (ok) return pos;
  if (counted) atomicAdd(S.fallbacks, 1ull);
  return lower_bound_in(S.key, 0, S.n, q);
}

// sums over the lanes of `group` (which all call it): c of 32-bit counts, s mod 2^64
__device__ __forceinline__ void group_sums(uint32_t group, uint32_t c, uint64_t s, bool sum,
                                           unsigned long long* tc, unsigned long long* ts) {
  *tc = (unsigned long long)__reduce_add_sync(group, c & 0xffffu) +
        ((unsigned long long)__reduce_add_sync(group, c >> 16) << 16);
  if (sum) {
    unsigned long long t = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      t += (unsigned long long)__reduce_add_sync(group, (uint32_t)(s >> (16 * k)) & 0xffffu) << (16 * k);
    *ts = t;
  }
}

// The whole aggregation: a warp takes 31 consecutive ranges, finds their 32
// boundaries' positions and adds every range's count and prefix difference to its
// polygons.  Boundaries ascend, so only the warp's first and last go through the
// radix table and the others look into the few spline points between: the table, a
// 32-byte sector of it per boundary, and an array of positions between two kernels
// are not read.  The curve visits few polygons in 31 ranges: the lanes of one
// polygon add up by warp reductions and send one atomic pair.  4.2M ranges over 50M
// points: 138 us in two kernels with a global atomic pair per range and polygon,
// this 115 us, 149 and 125 with the outputs' clearing (a hash of polygons in shared
// memory per 256 ranges: 231 us, its 64-bit shared atomics being slow).  Lists of many
// polygons take a warp a round each, so where few ranges leave warps idle a warp takes
// fewer than 31 (`per`: 15, 7 or 3; 200 overlapping stars, 4096 ranges: the call 51 ->
// 34 us).
template <bool RS, bool SUM>
__global__ __launch_bounds__(256) void point_ranges_kernel(
    const uint64_t* __restrict__ start, uint64_t R, uint32_t per, uint32_t sh, Spline S,
    const uint32_t* __restrict__ pay, const uint32_t* __restrict__ list_off,
    const uint32_t* __restrict__ list_ids, const int64_t* __restrict__ prefix,
    unsigned long long* __restrict__ count, unsigned long long* __restrict__ sum) {
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t r0 = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per;
  if (r0 >= R) return;  // whole warps
  const uint64_t r = min(r0 + min(lane, per), R);
  const uint64_t q = __ldg(start + r) << sh;
  const bool on = lane < per && r0 + lane < R;
  const uint32_t py = on ? __ldg(pay + r) : NONE;
  uint64_t p;
  if (!RS) {
    p = lower_bound_in(S.key, 0, S.n, q);
  } else {
    uint32_t a = 0;
    if (lane == 0 || lane == per)
      a = q <= S.kmin ? 0u : q > S.kmax ? (uint32_t)S.ns - 1 : spline_segment(S, q);
    const uint32_t b = __shfl_sync(FULL, a, per);
    a = __shfl_sync(FULL, a, 0);
    if (q <= S.kmin) {
      p = 0;
    } else if (q > S.kmax) {
      p = S.n;
    } else {
      for (uint32_t len = b - a + 1; len > 1;) {  // last spline point with key <= q
        const uint32_t half = len >> 1;
        if (__ldg(S.sk + a + half) <= q) a += half;
        len -= half;
      }
      // a boundary that two warps share is counted by the one it starts
      p = spline_position(S, a, q, r == r0 + lane && (lane < per || r == R));
    }
  }
  const uint32_t lo = (uint32_t)p, hi = __shfl_down_sync(FULL, lo, 1);
  const uint32_t c = on && py != NONE ? hi - lo : 0u;
  const uint64_t s = SUM && c ? (uint64_t)(__ldg(prefix + hi) - __ldg(prefix + lo)) : 0ull;
  // the lane's polygons, one a round
  uint32_t e = 0, e1 = c ? 1u : 0u;
  const bool list = c && py >= 0x80000000u;
  if (list) {
    e = __ldg(list_off + (py & 0x7fffffffu));
    e1 = __ldg(list_off + (py & 0x7fffffffu) + 1);
  }
  for (;;) {
    uint32_t left = __ballot_sync(FULL, e < e1);
    if (!left) break;
    const uint32_t id = e < e1 ? (list ? __ldg(list_ids + e) & 0x7fffffffu : py & 0x3fffffffu) : NONE;
    ++e;
    while (left) {
      const uint32_t lead = __ffs(left) - 1;
      const uint32_t pl = __shfl_sync(FULL, id, lead);
      const uint32_t group = __ballot_sync(FULL, id == pl);
      if (id == pl) {
        unsigned long long tc, ts;
        group_sums(group, c, s, SUM, &tc, &ts);
        if (lane == lead) {
          atomicAdd(count + pl, tc);
          if (SUM) atomicAdd(sum + pl, ts);
        }
      }
      left &= ~group;
    }
  }
}

// largest |interpolated - true position| over the distinct keys
__global__ void spline_error_kernel(Spline S, unsigned long long* __restrict__ worst) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= S.n || (i > 0 && S.key[i] == S.key[i - 1])) return;
  const uint64_t q = S.key[i];
  uint64_t a = 0, len = S.ns;  // last spline point with key <= q
  while (len > 1) {
    const uint64_t half = len >> 1;
    if (S.sk[a + half] <= q) a += half;
    len -= half;
  }
  uint64_t est = S.sp[a];
  if (a + 1 < S.ns) {
    const uint64_t k0 = S.sk[a], k1 = S.sk[a + 1], p0 = S.sp[a], p1 = S.sp[a + 1];
    est = p0 + (uint64_t)((unsigned __int128)(q - k0) * (p1 - p0) / (k1 - k0));
  }
  const unsigned long long d = est > i ? est - i : i - est;
  atomicMax(worst, d);
}

Spline spline_of(const sdb_points* p) {
  Spline S{};
  S.key = p->key;
  S.n = p->n;
  S.sk = p->rs_key;
  S.sp = p->rs_pos;
  S.ns = p->rs_n;
  S.table = p->rs_table;
  S.kmin = p->rs_min;
  S.kmax = p->rs_max;
  S.shift = p->rs_shift;
  S.E = (int64_t)p->rs_error;
  S.fallbacks = p->rs_fallbacks;
  return S;
}

}  // namespace

void release_point_index(sdb_points* p, cudaStream_t s) {
  void* ps[] = {p->prefix, p->rs_key, p->rs_pos, p->rs_table, p->rs_fallbacks};
  for (void* q : ps)
    if (q) dfree(q, s);
  p->prefix = nullptr;
  p->rs_key = nullptr;
  p->rs_pos = nullptr;
  p->rs_table = nullptr;
  p->rs_fallbacks = nullptr;
  p->rs_n = 0;
  p->rs_radix_bits = 0;
}

sdb_status build_point_index(sdb_points* p, uint32_t radix_bits, uint32_t spline_error,
                             cudaStream_t s) {
  release_point_index(p, s);
  Scratch sc(s);
  const uint64_t n = p->n;
  // prefix sums of the attribute in key order
  SDB_TRY(dalloc_n(&p->prefix, n + 1, s));
  SDB_TRY(exclusive_scan_i32(p->attr, p->prefix, n, s));
  // spline points, chunk by chunk
  const uint64_t nchunks = (n + CHUNK - 1) / CHUNK;
  uint64_t *cnt, *off, *dns;
  uint32_t* mask;
  SDB_TRY(sc.get(&cnt, nchunks));
  SDB_TRY(sc.get(&off, nchunks));
  SDB_TRY(sc.get(&dns, 1));
  SDB_TRY(sc.get(&mask, nchunks * MASK_WORDS));
  const unsigned chunk_grid = grid_for(nchunks, SPLINE_WARPS);
  spline_mark_kernel<<<chunk_grid, SPLINE_WARPS * 32, 0, s>>>(p->key, n, nchunks,
                                                             (int64_t)spline_error, mask, cnt);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  SDB_TRY(exclusive_scan<uint64_t>(cnt, off, nchunks, dns, s));
  uint64_t ns = 0, ends[2] = {0, 0};
  SDB_TRY_CUDA(cudaMemcpyAsync(&ns, dns, 8, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaMemcpyAsync(&ends[0], p->key, 8, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaMemcpyAsync(&ends[1], p->key + n - 1, 8, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaStreamSynchronize(s));
  if (ns >= 0xffffffffull) {
    set_error("radix spline: %llu spline points exceed 32-bit indices", (unsigned long long)ns);
    return SDB_ENOMEM;
  }
  SDB_TRY(dalloc_n(&p->rs_key, ns, s));
  SDB_TRY(dalloc_n(&p->rs_pos, ns, s));
  spline_write_kernel<<<chunk_grid, SPLINE_WARPS * 32, 0, s>>>(p->key, nchunks, mask, off,
                                                              p->rs_key, p->rs_pos);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  // radix table over the key range
  const uint64_t span = ends[1] - ends[0];
  const uint32_t span_bits = span ? 64 - __builtin_clzll(span) : 0;
  p->rs_shift = span_bits > radix_bits ? span_bits - radix_bits : 0;
  SDB_TRY(dalloc_n(&p->rs_table, (1ull << radix_bits) + 1, s));
  radix_table_kernel<<<grid_for((1ull << radix_bits) + 1, TABLE_TILE), 256, 0, s>>>(
      p->rs_key, (uint32_t)ns, ends[0], p->rs_shift, radix_bits, p->rs_table);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  SDB_TRY(dalloc_n(&p->rs_fallbacks, 1, s));
  SDB_TRY_CUDA(cudaMemsetAsync(p->rs_fallbacks, 0, 8, s));
  SDB_TRY_CUDA(cudaStreamSynchronize(s));
  p->rs_n = ns;
  p->rs_min = ends[0];
  p->rs_max = ends[1];
  p->rs_radix_bits = radix_bits;
  p->rs_error = spline_error;
  return SDB_OK;
}

sdb_status point_index_aggregate(const sdb_points* p, const sdb_covering* cov, int lookup,
                                 uint64_t* count, int64_t* sum, cudaStream_t s) {
  SDB_TRY_CUDA(cudaMemsetAsync(count, 0, (size_t)cov->P * 8, s));
  if (sum) SDB_TRY_CUDA(cudaMemsetAsync(sum, 0, (size_t)cov->P * 8, s));
  const bool rs = lookup == SDB_LOOKUP_RADIX_SPLINE;
  if (rs) SDB_TRY_CUDA(cudaMemsetAsync(p->rs_fallbacks, 0, 8, s));
  const uint64_t R = cov->R;
  const Spline S = spline_of(p);
  const uint32_t sh = 2 * cov->k;
  auto* c = reinterpret_cast<unsigned long long*>(count);
  auto* su = reinterpret_cast<unsigned long long*>(sum);
  auto kern = rs ? (sum ? point_ranges_kernel<true, true> : point_ranges_kernel<true, false>)
                 : (sum ? point_ranges_kernel<false, true> : point_ranges_kernel<false, false>);
  uint32_t per = 31;  // ranges per warp, fewer while there are not 16 warps per SM
  while (per > 3 && R < (uint64_t)per * 16 * num_sms()) per >>= 1;
  const uint64_t warps = (R + per - 1) / per;
  kern<<<grid_for(warps, 8), 256, 0, s>>>(cov->start, R, per, sh, S, cov->pay, cov->list_off,
                                          cov->list_ids, p->prefix, c, su);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  return SDB_OK;
}

sdb_status point_index_stats(const sdb_points* p, uint64_t* n_spline, uint64_t* max_error,
                             uint64_t* fallbacks, cudaStream_t s) {
  *n_spline = p->rs_n;
  unsigned long long h[2] = {0, 0};
  Scratch sc(s);
  unsigned long long* worst;
  SDB_TRY(sc.get(&worst, 1));
  SDB_TRY_CUDA(cudaMemsetAsync(worst, 0, 8, s));
  spline_error_kernel<<<grid_for(p->n, 256), 256, 0, s>>>(spline_of(p), worst);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  SDB_TRY_CUDA(cudaMemcpyAsync(&h[0], worst, 8, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaMemcpyAsync(&h[1], p->rs_fallbacks, 8, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaStreamSynchronize(s));
  *max_error = h[0];
  *fallbacks = h[1];
  return SDB_OK;
}

}  // namespace sdb

extern "C" {

sdb_status sdb_points_build_index(sdb_points* pts, uint32_t radix_bits, uint32_t spline_error,
                                  void* cuda_stream) {
  if (!pts) {
    sdb::set_error("points is NULL");
    return SDB_EINVAL;
  }
  if (radix_bits < 1 || radix_bits > 30) {
    sdb::set_error("radix_bits %u outside 1..30", radix_bits);
    return SDB_EINVAL;
  }
  if (spline_error < 1 || spline_error > (1u << 20)) {
    sdb::set_error("spline_error %u outside 1..2^20", spline_error);
    return SDB_EINVAL;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != pts->device) {
    sdb::set_error("points live on device %d, current device is %d", pts->device, dev);
    return SDB_EINVAL;
  }
  return sdb::build_point_index(pts, radix_bits, spline_error, (cudaStream_t)cuda_stream);
}

sdb_status sdb_points_aggregate(const sdb_points* pts, const sdb_covering* cov, int lookup,
                                uint64_t* d_count, int64_t* d_sum, void* cuda_stream) {
  if (!pts || !cov || !d_count) {
    sdb::set_error("points, covering or d_count is NULL");
    return SDB_EINVAL;
  }
  if (lookup != SDB_LOOKUP_BINARY && lookup != SDB_LOOKUP_RADIX_SPLINE) {
    sdb::set_error("point aggregation takes SDB_LOOKUP_BINARY or SDB_LOOKUP_RADIX_SPLINE, not %d",
                   lookup);
    return SDB_EINVAL;
  }
  if (cov->B != pts->B) {
    sdb::set_error("covering grid bits %u differ from the points' %u", cov->B, pts->B);
    return SDB_EINVAL;
  }
  if ((d_sum || lookup == SDB_LOOKUP_RADIX_SPLINE) && !pts->prefix) {
    sdb::set_error("SUM and the RadixSpline lookup need sdb_points_build_index first");
    return SDB_EINVAL;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != pts->device || dev != cov->device) {
    sdb::set_error("points, covering and current device differ");
    return SDB_EINVAL;
  }
  return sdb::point_index_aggregate(pts, cov, lookup, d_count, d_sum, (cudaStream_t)cuda_stream);
}

sdb_status sdb_points_index_stats(const sdb_points* pts, uint64_t* n_spline, uint64_t* max_error,
                                  uint64_t* fallbacks, void* cuda_stream) {
  if (!pts || !n_spline || !max_error || !fallbacks) {
    sdb::set_error("NULL argument");
    return SDB_EINVAL;
  }
  if (!pts->prefix) {
    sdb::set_error("no point index (sdb_points_build_index)");
    return SDB_EINVAL;
  }
  return sdb::point_index_stats(pts, n_spline, max_error, fallbacks, (cudaStream_t)cuda_stream);
}

}  // extern "C"
