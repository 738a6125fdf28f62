// Learned range index over the covering's sorted range starts (Sec. 3, "Point
// Indexing": learning the position of a key in the sorted array to speed up the
// search; RadixSpline is the paper's model, a two-level piecewise-linear model
// is used here).
//
//   root:  leaf(h) = clamp(floor(knot_j + (knot_{j+1} - knot_j) * frac), 0, L-1)  (FP32)
//          with j = h >> wshift, frac = (h - (j << wshift)) / 2^wshift and
//          knot_j = L * #{i : start_i < j << wshift} / R  (2^K uniform knots,
//          K = 12 by default; K = 0 is a single root line over [0, 4^F))
//   leaf:  pred(h) = first + floor(fma(a, float(h - base), b))         (FP32)
//
// Both maps are monotone in h.  The root is the piecewise-linear interpolant of
// the range starts' cumulative distribution, so leaves receive roughly equal
// numbers of ranges even where ranges crowd along polygon boundaries (a single
// line through (start_i, i) routes most ranges to a few leaves: the covering's
// id -> index map is a staircase at every scale).  Leaf l receives exactly the ids h in
// [base_l, base_{l+1}), where base_l is the smallest id the root sends to a
// leaf >= l; it is found by binary search on the root function itself, with the
// same instructions the lookup uses, so routing at fit time and lookup time
// agree bit for bit.  By monotonicity start_i < base_l exactly when the root
// sends start_i to a leaf below l, so one pass over the ranges counts the
// starts below every leaf's base, which fixes each leaf's first and last range.  The leaf line is a least-squares fit of the range index
// (relative to the leaf's first range) on the leaf-relative id.  Its error
// window covers, for every range i the leaf can see, every id of
// [start_i, start_{i+1}) that the leaf receives: by monotonicity it is enough to
// evaluate the prediction at the two ends of each such interval.  Lookups are
// verified anyway and fall back to binary search.
#include "sdb_internal.cuh"

namespace sdb {

namespace {

constexpr unsigned FULL = 0xffffffffu;
// knot j: L * (number of range starts below j << wshift) / R
__global__ void knots_kernel(const uint64_t* __restrict__ start, uint64_t R, uint32_t K,
                             uint32_t wshift, uint32_t L, float* __restrict__ knot) {
  uint32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j > K) return;
  const uint64_t key = (uint64_t)j << wshift;
  uint64_t lo = 0, len = R;  // first i with start[i] >= key
  while (len > 0) {
    uint64_t half = len >> 1;
    if (start[lo + half] < key) {
      lo += half + 1;
      len -= half + 1;
    } else {
      len = half;
    }
  }
  knot[j] = (float)((double)L * (double)lo / (double)R);
}

// base of every leaf l in [0, L]: smallest h in [0, top] with leaf(h) >= l
__global__ void leaf_base_kernel(const float* __restrict__ knot, uint32_t wshift, float inv_w,
                                 uint32_t L, uint64_t top, uint64_t* __restrict__ base) {
  uint32_t l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l > L) return;
  if (l == 0) {
    base[0] = 0;
    return;
  }
  if (l == L) {
    base[L] = top;
    return;
  }
  uint64_t lo = 0, hi = top;
  while (lo < hi) {
    uint64_t mid = lo + ((hi - lo) >> 1);
    if (root_leaf(knot, wshift, inv_w, L, mid) >= l)
      hi = mid;
    else
      lo = mid + 1;
  }
  base[l] = lo;
}

// fence j: the range start of index j << FENCE_SHIFT (j <= R >> FENCE_SHIFT)
__global__ void fence_kernel(const uint64_t* __restrict__ start, uint64_t nf,
                             uint64_t* __restrict__ fence) {
  const uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j < nf) fence[j] = start[j << FENCE_SHIFT];
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

__device__ __forceinline__ long long warp_max(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    long long t = __shfl_xor_sync(FULL, v, o);
    v = t > v ? t : v;
  }
  return v;
}

// below[l] = #{i < R : start_i < base_l} for l in [0, L].  Range i's start
// goes to leaf lam_i; the leaves lam_{i-1} < l <= lam_i have exactly i starts
// below their base (lam_{-1} = -1, and start_R = 4^F stands for leaf L).  A thread's
// work is one chain of dependent reads: BELOW_ITEMS starts per thread, all read first
// (263-zone sweep, 27M ranges: 122 us with one, 101 with four).  One start per thread
// where leaves outnumber ranges: the leaves between two starts are then the longer chain
// (2^20 leaves over 4^8 ids, the whole index: 670 us with four, 440 with one).
template <int BELOW_ITEMS>
__global__ void leaf_below_kernel(const uint64_t* __restrict__ start, uint64_t R,
                                  const float* __restrict__ knot, uint32_t wshift, float inv_w,
                                  uint32_t L, uint32_t* __restrict__ below) {
  const uint64_t i0 = (uint64_t)blockIdx.x * BELOW_ITEMS * blockDim.x + threadIdx.x;
  uint64_t at[BELOW_ITEMS], before[BELOW_ITEMS];
#pragma unroll
  for (int j = 0; j < BELOW_ITEMS; ++j) {
    const uint64_t i = i0 + j * blockDim.x;
    at[j] = i <= R ? start[i] : 0ull;
    before[j] = i > 0 && i <= R ? start[i - 1] : 0ull;
  }
#pragma unroll
  for (int j = 0; j < BELOW_ITEMS; ++j) {
    const uint64_t i = i0 + j * blockDim.x;
    if (i > R) return;
    const uint32_t lam = i < R ? root_leaf(knot, wshift, inv_w, L, at[j]) : L;
    const uint32_t from = i == 0 ? 0u : root_leaf(knot, wshift, inv_w, L, before[j]) + 1u;
    for (uint32_t l = from; l <= lam; ++l) below[l] = (uint32_t)i;
  }
}

__device__ __forceinline__ float to_float(uint32_t v) { return __uint2float_rn(v); }
__device__ __forceinline__ float to_float(uint64_t v) { return __ull2float_rn(v); }
__device__ __forceinline__ void to_floor(float v, int32_t* o) { *o = __float2int_rd(v); }
__device__ __forceinline__ void to_floor(float v, int64_t* o) { *o = __float2ll_rd(v); }

// The line and window of the leaf [b0, b1) over the ranges [first, first + n).  Bound
// by the conversions between integers and FP32: a leaf narrower than 2^32 ids holds
// fewer ranges than that, and 32-bit integers give the same floats and the same clamped
// positions as 64-bit ones (U unsigned, S signed) in 207 instead of 614 us for the
// 263-zone sweep's 27M ranges.  (Four loads in flight per lane changed nothing: 623.)
template <class U, class S>
__device__ __forceinline__ void fit_leaf(const uint64_t* __restrict__ start, uint64_t first,
                                         uint64_t n, uint64_t b0, uint64_t b1, LeafRec* lr,
                                         long long* lo, long long* hi) {
  const U nn = (U)n;
  const uint64_t* __restrict__ s = start + first;
  // pass 1: means; pass 2: centred moments (FP32: the fit only shapes the
  // windows, which come from the lookup's own arithmetic in pass 3)
  float sx = 0.f, sy = 0.f;
  for (U i = threadIdx.x & 31; i < nn; i += 32) {
    sx += to_float((U)((s[i] > b0 ? s[i] : b0) - b0));
    sy += to_float(i);
  }
  const float inv_n = 1.0f / to_float(nn);
  const float mx = warp_sum(sx) * inv_n, my = warp_sum(sy) * inv_n;
  float sxx = 0.f, sxy = 0.f;
  for (U i = threadIdx.x & 31; i < nn; i += 32) {
    const float dx = to_float((U)((s[i] > b0 ? s[i] : b0) - b0)) - mx, dy = to_float(i) - my;
    sxx = fmaf(dx, dx, sxx);
    sxy = fmaf(dx, dy, sxy);
  }
  sxx = warp_sum(sxx);
  sxy = warp_sum(sxy);
  const float slope = (sxx > 0.f && sxy > 0.f) ? sxy / sxx : 0.f;
  lr->a = slope;
  lr->b = my - slope * mx;
  // pass 3: error window with the lookup's own FP32 arithmetic (leaf_predict,
  // positions counted from the leaf's first)
  auto predict = [&](U x) {
    S p;
    to_floor(__fmaf_rn(lr->a, to_float(x), lr->b), &p);
    p = p < 0 ? 0 : p;
    return p > (S)(nn - 1) ? (S)(nn - 1) : p;
  };
  S ehi = 0, elo = 0;
  for (U i = threadIdx.x & 31; i < nn; i += 32) {
    const uint64_t lo_h = s[i] > b0 ? s[i] : b0, hi_h = (s[i + 1] < b1 ? s[i + 1] : b1) - 1;
    const S up = (S)i - predict((U)(lo_h - b0)), dn = predict((U)(hi_h - b0)) - (S)i;
    ehi = up > ehi ? up : ehi;
    elo = dn > elo ? dn : elo;
  }
  *hi = warp_max(ehi);
  *lo = warp_max(elo);
}

// PER leaves per warp: a lane looks at each, writes it if no id is routed to it or one
// range holds all of its ids (the constant line, without error), and the warp fits the
// others one after the other: centred least squares (FP32), error window.  One leaf per
// warp, or 32 where leaves outnumber ranges, few are fitted and 4096 warps are left (2^20
// leaves over 4^8 ids, the whole index: 440 -> 290 us; 250,000 ranges: 720 -> 300).
template <int PER>
__global__ __launch_bounds__(256, 6) void leaf_fit_kernel(const uint64_t* __restrict__ start,
                                                          uint64_t R,
                                                          const uint64_t* __restrict__ base,
                                                          const uint32_t* __restrict__ below,
                                                          uint32_t L, LeafRec* __restrict__ leaves) {
  const uint32_t l0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * PER;
  const int lane = threadIdx.x & 31;
  if (l0 >= L) return;  // whole warps (L is a multiple of PER)
  uint64_t b0 = 0, b1 = 0, first = 0, last = 0;
  bool fit = false;
  if (lane < PER) {
    const uint32_t l = l0 + lane;
    b0 = base[l];
    b1 = base[l + 1];
    // range holding b0: the last start <= b0 (b0 < 4^F = start[R] for l < L)
    const uint32_t c0 = below[l];
    first = (c0 < R && start[c0] == b0) ? c0 : (uint64_t)c0 - 1;
    first = first < R ? first : R - 1;
    last = first;
    if (b0 < b1) {
      last = (uint64_t)below[l + 1] - 1;  // range holding b1 - 1
      last = last < first ? first : (last < R ? last : R - 1);
    }
    fit = last > first;
    if (!fit) leaves[l] = LeafRec{b0, 0.f, 0.f, (uint32_t)first, (uint32_t)last, 0, 0};
  }
  for (uint32_t todo = __ballot_sync(0xffffffffu, fit); todo; todo &= todo - 1) {
    const int j = __ffs(todo) - 1;
    const uint64_t B0 = __shfl_sync(0xffffffffu, (unsigned long long)b0, j);
    const uint64_t B1 = __shfl_sync(0xffffffffu, (unsigned long long)b1, j);
    const uint64_t f = __shfl_sync(0xffffffffu, (unsigned long long)first, j);
    const uint64_t n = __shfl_sync(0xffffffffu, (unsigned long long)last, j) - f + 1;
    LeafRec lr{B0, 0.f, 0.f, (uint32_t)f, (uint32_t)(f + n - 1), 0, 0};
    long long ehi = 0, elo = 0;
    if (B1 - B0 <= 0xffffffffull)
      fit_leaf<uint32_t, int32_t>(start, f, n, B0, B1, &lr, &elo, &ehi);
    else
      fit_leaf<uint64_t, int64_t>(start, f, n, B0, B1, &lr, &elo, &ehi);
    const long long CAP = 1ll << 30;
    lr.errhi = (int32_t)(ehi > CAP ? CAP : ehi);
    lr.errlo = (int32_t)(elo > CAP ? CAP : elo);
    if (lane == 0) leaves[l0 + j] = lr;
  }
}

}  // namespace

sdb_status build_learned_index(sdb_covering* cov, uint32_t leaf_bits, uint32_t root_bits,
                               cudaStream_t s) {
  TraceScope tr("index.build", s);
  const uint32_t L = 1u << leaf_bits;
  const uint64_t R = cov->R;
  const uint64_t top = 1ull << (2 * cov->F);
  const uint32_t kbits = 2 * cov->F < root_bits ? 2 * cov->F : root_bits;
  const uint32_t K = 1u << kbits;
  const uint32_t wshift = 2 * cov->F - kbits;
  const float inv_w = 1.0f / (float)(1ull << wshift);  // exact: a power of two
  Scratch sc(s);
  if (cov->leaves) dfree(cov->leaves, s);
  if (cov->knots) dfree(cov->knots, s);
  if (cov->fence) dfree(cov->fence, s);
  cov->leaves = nullptr;
  cov->knots = nullptr;
  cov->fence = nullptr;
  const uint64_t nf = (R >> FENCE_SHIFT) + 1;
  SDB_TRY(dalloc_n(&cov->fence, nf, s));
  fence_kernel<<<grid_for(nf, 256), 256, 0, s>>>(cov->start, nf, cov->fence);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  SDB_TRY(dalloc_n(&cov->leaves, L, s));
  if (reinterpret_cast<uintptr_t>(cov->leaves) & 31u) {  // the lookup reads 32 bytes at once
    set_error("learned index: leaf records not 32-byte aligned");
    return SDB_ECUDA;
  }
  SDB_TRY(dalloc_n(&cov->knots, (size_t)K + 1, s));
  if (!cov->fallbacks) {
    SDB_TRY(dalloc_n(&cov->fallbacks, 1, s));
    SDB_TRY_CUDA(cudaMemsetAsync(cov->fallbacks, 0, sizeof(unsigned long long), s));
  }
  knots_kernel<<<grid_for((size_t)K + 1, 256), 256, 0, s>>>(cov->start, R, K, wshift, L, cov->knots);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  uint64_t* base;
  uint32_t* below;
  SDB_TRY(sc.get(&base, (size_t)L + 1));
  SDB_TRY(sc.get(&below, (size_t)L + 1));
  leaf_base_kernel<<<grid_for((size_t)L + 1, 256), 256, 0, s>>>(cov->knots, wshift, inv_w, L, top,
                                                                 base);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  if (R > L)
    leaf_below_kernel<4><<<grid_for((size_t)R + 1, 256 * 4), 256, 0, s>>>(cov->start, R, cov->knots,
                                                                          wshift, inv_w, L, below);
  else
    leaf_below_kernel<1><<<grid_for((size_t)R + 1, 256), 256, 0, s>>>(cov->start, R, cov->knots,
                                                                      wshift, inv_w, L, below);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  if (R > L || L < (1u << 17))
    leaf_fit_kernel<1><<<grid_for((size_t)L * 32, 256), 256, 0, s>>>(cov->start, R, base, below, L,
                                                                     cov->leaves);
  else
    leaf_fit_kernel<32><<<grid_for(L, 256), 256, 0, s>>>(cov->start, R, base, below, L,
                                                         cov->leaves);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  SDB_TRY_CUDA(cudaStreamSynchronize(s));
  cov->leaf_bits = leaf_bits;
  cov->knot_bits = kbits;
  cov->knot_wshift = wshift;
  return SDB_OK;
}

}  // namespace sdb
