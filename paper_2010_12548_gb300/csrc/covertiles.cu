// Covering tiles: the last TILE_DEPTH levels of the covering's refinement, done
// as bitmaps instead of cell by cell.
//
// The level-synchronous refinement (cover.cu) stops TILE_DEPTH levels above a
// query's finest level.  What it has produced by then -- interior cells of the
// coarser levels and boundary cells ("tiles" of 32 x 32 finest cells, each with
// the polygon's edges that meet it and the parity of its corner) -- is about a
// fiftieth of the finest covering, and only that is sorted by (query, curve
// position).  A covering then needs, per tile and polygon, which of the 1024
// finest cells belong to it:
//   * a cell that an edge touches does (closed cell, closed edge).  Lane = row of
//     the tile; the edge clipped to the row's closed strip covers one run of
//     cells, found exactly: the column at which the edge's line meets a row line is
//     a quotient of at most 32, estimated in FP32 and settled by its remainder.
//   * an untouched cell does when its corner is inside: the tile corner's parity
//     and the crossings from there up the left side and along the row's line,
//     decided with the refinement's symbolic perturbation (cover.cu).
// The 32 row words become 32 words in curve order (bit t of the tile = curve
// position t).  There a quadtree cell of level l is an aligned run of 4^l bits,
// so the covering's records (maximal untouched cells, and the viewport clip that
// keeps or drops a record as a whole) and the starts of the canonical ranges
// (positions where a polygon's bit changes) are shifts and masks of whole words.
// Ranges are written from the bitmaps directly: no record of a finest cell is
// ever stored, sorted or merged.
//
// One warp per tile, a block where more than CROWD polygons meet.  For the 263-zone
// sweep (eps 2^12 .. 2^6, 1.2e8 records) this stage takes 2.64 ms traced (raster 1.28,
// ranges 0.65, sort 0.29, elements, groups and waits)
// where the refinement to the finest level, its sort and its merge took 9.3
// (2.4, 4.5 and 2.2, and the counters of five more levels).
#include "cover_internal.cuh"

#include <algorithm>
#include <string>
#include <vector>

namespace sdb {

namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr uint32_t NONE = 0xffffffffu;
constexpr int TPB = 256;
constexpr int WPB = TPB / 32;
// counters that a sum over all tiles, and one over all blocks, is spread over
constexpr uint32_t FRONT_SPREAD = 256, SPREAD = 64;

// element info: slot (bits 0..25), covers the group's first cell (26), with the
// boundary flag (27), covers its last cell (28), with the flag (29), tile (30)
constexpr uint32_t INFO_SLOT = (1u << 26) - 1u;
constexpr uint32_t INFO_FIRST = 26, INFO_LAST = 28, INFO_TILE = 1u << 30;

// ---------------------------------------------------------------- rasterising
// floor(f / d) for d > 0 where it lies in [-2, 34], else some value on the same
// side of that interval; *exact: f is a multiple of d.  rd is about 1 / d: the
// estimate is within one, the remainder decides.
__device__ __forceinline__ int column_of(int64_t f, int64_t d, float rd, bool* exact) {
  const float q = fminf(fmaxf(__ll2float_rn(f) * rd, -2.0f), 34.0f);
  int t = (int)floorf(q);
  int64_t r = f - (int64_t)t * d;
  if (r < 0) {
    --t;
    r += d;
  } else if (r >= d) {
    ++t;
    r -= d;
  }
  *exact = r == 0;
  return t;
}

// Row words of one polygon in one tile (lane = row, bit = column): *touched the
// cells that an edge meets, *inside the untouched cells in the polygon.  px, py
// is the tile's corner, sh the finest cells' side (log2), par the parity of the
// perturbed corner.  All lanes take part.
//
// For an edge from a up to b, f(row) = cross(b - a, (px, Y0) - a) over dy side is
// the column at which the edge's line meets the row's lower line: one exact small
// quotient per row, whose remainder tells whether a column line is met exactly.
__device__ __forceinline__ void raster_tile(const Edge* __restrict__ edges,
                                            const uint32_t* __restrict__ elist, uint32_t ecnt,
                                            int32_t px, int32_t py, uint32_t sh, uint32_t par,
                                            uint32_t* touched, uint32_t* inside) {
  const int lane = threadIdx.x & 31;
  const int32_t s = 1 << sh;
  const int32_t Y0 = py + lane * s, Y1 = Y0 + s;  // the row's closed strip
  uint32_t T = 0, H = 0, V = 0;  // touched; flips along the row; flip of the row's corner
  for (uint32_t base = 0; base < ecnt; base += 32) {
    Edge E{0, 0, 0, 0};
    if (base + lane < ecnt) {
      E = edges[__ldg(elist + base + lane)];
      if (E.by < E.ay) E = Edge{E.bx, E.by, E.ax, E.ay};  // upwards
    }
    const int m = (int)min(32u, ecnt - base);
    for (int e = 0; e < m; ++e) {
      const int32_t ax = __shfl_sync(FULL, E.ax, e), ay = __shfl_sync(FULL, E.ay, e);
      const int32_t bx = __shfl_sync(FULL, E.bx, e), by = __shfl_sync(FULL, E.by, e);
      const int32_t dx = bx - ax, dy = by - ay;
      const int64_t d = (int64_t)dy << sh, step = (int64_t)dx << sh;
      const int64_t f0 = (int64_t)dx * (py - ay) - (int64_t)dy * (px - ax);
      const int64_t f = f0 + lane * step;
      const float rd = dy > 0 ? __frcp_rn(__ll2float_rn(d)) : 0.0f;
      bool exl, exu, ex32;
      const int tl = column_of(f, d, rd, &exl);
      int tu = __shfl_down_sync(FULL, tl, 1);
      exu = __shfl_down_sync(FULL, (int)exl, 1) != 0;
      const int t32 = column_of(f0 + 32 * step, d, rd, &ex32);  // the tile's upper line
      if (lane == 31) {
        tu = t32;
        exu = ex32;
      }
      // the clipped edge's ends by column: where it leaves the strip, or its own
      // end inside it (a horizontal edge always has both ends inside)
      const bool cut_lo = Y0 > ay, cut_hi = Y1 < by;
      const int t_lo = cut_lo ? tl : (ax - px) >> sh, t_hi = cut_hi ? tu : (bx - px) >> sh;
      const bool e_lo = cut_lo ? exl : ((ax - px) & (s - 1)) == 0;
      const bool e_hi = cut_hi ? exu : ((bx - px) & (s - 1)) == 0;
      // closed cells: one more to the left when the left end is on a column line
      const int m0 = dx >= 0 ? t_lo - e_lo : t_hi - e_hi, m1 = dx >= 0 ? t_hi : t_lo;
      if (by >= Y0 && ay <= Y1 && m1 >= 0 && m0 <= 31)
        T |= (FULL << max(m0, 0)) & (FULL >> (31 - min(m1, 31)));
      // perturbed side of the row's left corner, and of the tile's
      const bool tie = dy == 0 && dx > 0;
      const bool pos = f > 0 || (f == 0 && tie), pos0 = f0 > 0 || (f0 == 0 && tie);
      if ((ax > px) != (bx > px)) V ^= (uint32_t)(pos != pos0);
      // the edge crosses the row's line right of that corner: every later corner flips
      if (ay <= Y0 && by > Y0 && pos && tl < 31) H ^= FULL << (tl + 1);
    }
  }
  *touched = T;
  *inside = (((par ^ V) & 1u) ? ~H : H) & ~T;
}

// ---------------------------------------------------------------- curve order
// The tile's curve by 2 x 2 blocks: lane l holds curve positions 32 l .. 32 l + 31,
// the blocks 8 l .. 8 l + 7 of the curve over 16 x 16 blocks.  s_blk[i * 32 + l]
// describes block 8 l + i in the plain orientation -- bits 0..6 the byte offset of
// its two row words (8 by), bits 8..12 its first column (2 bx), bits 16..21 its
// own orientation times 16 -- and s_blk[256 + ...] the same with x and y swapped;
// complementing is an XOR of the fields.  s_perm[orientation * 16 + v] puts a
// block's four cells v (bit 2 y + x) in curve order.
constexpr uint32_t BLK_COMPLEMENT = (15u << 3) | (15u << 9) | (1u << 20);
struct CurveTables {
  uint32_t blk[512];
  uint8_t perm[64];
};
__device__ __forceinline__ void fill_curve(CurveTables& t) {
  for (uint32_t k = threadIdx.x; k < 256; k += TPB) {
    uint32_t sw = 0, cm = 0, x = 0, y = 0;
    for (int lev = TILE_DEPTH - 2; lev >= 0; --lev) {
      const uint32_t d = (k >> (2 * lev)) & 3u;
      const uint32_t xt = d >> 1, yt = xt ^ (d & 1u);
      const uint32_t u = xt ^ cm, v = yt ^ cm;
      x = (x << 1) | (sw ? v : u);
      y = (y << 1) | (sw ? u : v);
      if (!yt) {
        sw ^= 1u;
        cm ^= xt;
      }
    }
    const uint32_t at = (k & 7u) * 32 + (k >> 3), o = (sw << 1) | cm;
    t.blk[at] = (y << 3) | (x << 9) | (o << 20);
    t.blk[256 + at] = (x << 3) | (y << 9) | ((o ^ 2u) << 20);
  }
  for (uint32_t k = threadIdx.x; k < 64; k += TPB) {
    const uint32_t sw = k >> 5, cm = (k >> 4) & 1u;
    uint32_t out = 0;
    for (uint32_t d = 0; d < 4; ++d) {
      const uint32_t xt = d >> 1, yt = xt ^ (d & 1u);
      const uint32_t u = xt ^ cm, v = yt ^ cm;
      const uint32_t x = sw ? v : u, y = sw ? u : v;
      out |= ((k >> (2 * y + x)) & 1u) << d;
    }
    t.perm[k] = (uint8_t)out;
  }
}

// N row words (lane = row) to curve order (lane l: positions 32 l .. 32 l + 31)
// through shared memory, a 2 x 2 block at a time: one 8-byte read of its two
// rows, one read of the permutation.  (A bit at a time took 450 instructions for
// two words; this takes 190.)
template <int N>
__device__ __forceinline__ void to_curve(const uint32_t (&rows)[N], uint32_t (&out)[N],
                                         uint32_t orient, const CurveTables& t,
                                         uint32_t (*s_rows)[32]) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll
  for (int n = 0; n < N; ++n) s_rows[n][lane] = rows[n];
  __syncwarp();
  const uint32_t flip = (orient & 1u) ? BLK_COMPLEMENT : 0u;
  const uint32_t* blk = t.blk + ((orient & 2u) ? 256 : 0) + lane;
#pragma unroll
  for (int n = 0; n < N; ++n) out[n] = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t e = blk[i * 32] ^ flip;
    const uint32_t c = (e >> 8) & 31u;
    const uint8_t* perm = t.perm + ((e >> 16) & 0x30u);
#pragma unroll
    for (int n = 0; n < N; ++n) {
      const uint2 w = *reinterpret_cast<const uint2*>(
          reinterpret_cast<const unsigned char*>(s_rows[n]) + (e & 0x78u));
      const uint32_t v = ((w.x >> c) & 3u) | (((w.y >> c) & 3u) << 2);
      out[n] |= (uint32_t)perm[v] << (4 * i);
    }
  }
}

// per aligned run of 4, 16, 64, 256 bits: all ones if any bit of the run is set
__device__ __forceinline__ uint32_t any4(uint32_t v) {
  v |= v >> 1;
  v |= v >> 2;
  return (v & 0x11111111u) * 15u;
}
__device__ __forceinline__ uint32_t any16(uint32_t v) {
  return ((v & 0xffffu) ? 0xffffu : 0u) | ((v >> 16) ? 0xffff0000u : 0u);
}
__device__ __forceinline__ uint32_t any_lanes(uint32_t v, int lanes) {  // lanes = 2 or 8
  const uint32_t b = __ballot_sync(FULL, v != 0);
  const uint32_t g = (threadIdx.x & 31) & ~(uint32_t)(lanes - 1);
  return ((b >> g) & ((1u << lanes) - 1u)) ? FULL : 0u;
}

// What a warp needs of one polygon in one tile, in sorted order (32 bytes)
struct __align__(16) TileRec {
  int32_t px, py;     // the tile's corner
  uint32_t eoff, ecnt_par;
  uint32_t slot;
  uint32_t geo;       // finest side (log2) | orientation << 8 | clipped << 10
  uint32_t query;
  uint32_t bits;      // its bitmap's place (its tile item)
};

// The tile groups: first element and elements, in any order.  Those of more than CROWD
// polygons come last (from the array's end backwards): blocks raster them, not warps.
constexpr uint32_t CROWD = 8;
struct TileHeads {
  uint2* at;
  uint32_t* n;  // the groups of up to CROWD polygons, and the larger ones
  uint32_t cap;
  __device__ uint32_t all() const { return n[0] + n[1]; }
  __device__ uint2 operator[](uint32_t g) const {
    return g < n[0] ? at[g] : at[cap - 1 - (g - n[0])];
  }
};

struct TileArgs {
  const TileRec* rec;      // per element (tiles' only)
  const uint32_t* elist;
  const Edge* edges;
  const CoverQuery* qs;
  uint32_t qshift, flags;
  const uint64_t* key;     // sorted keys
  uint64_t ne;
  TileHeads heads;
  uint32_t* bits;          // per item 32 words in curve order: the polygon's cells
  uint32_t* bbits;         // the same for its boundary cells (flagged coverings)
  uint32_t* info;          // per element
  uint32_t* cells;         // per element: records of the group (at its head)
  uint64_t* inner;         // per element, at tile heads: ranges that start inside
                           // the tile << 32 | their list entries
  unsigned int* flag;      // [0] nested cells, [1] a tile with too many polygons,
                           // [2] polygons that overlap inside a tile
  unsigned long long* front;  // boundary cells one level above the finest
};

// What a tile's polygons add up to, per lane
struct TileSum {
  uint32_t starts = 0;  // positions where the set of polygons changes
  uint32_t cells = 0;   // records, in 256ths
  uint32_t front = 0;   // boundary cells one level above the finest
  uint32_t u[5] = {0, 0, 0, 0, 0};  // cells by the level of their record
};

// element i's polygon: its bitmaps, its info, what it adds to the tile
__device__ __forceinline__ void raster_element(const TileArgs& A, uint32_t i, uint32_t lane,
                                               const CurveTables& s_curve,
                                               uint32_t (*s_rows)[32], TileSum& S) {
  const TileRec R = A.rec[i];
  const uint32_t sh = R.geo & 0xffu, orient = (R.geo >> 8) & 3u;
  uint32_t rows[2], curve[2];
  raster_tile(A.edges, A.elist + R.eoff, R.ecnt_par & 0x7fffffffu, R.px, R.py, sh,
              R.ecnt_par >> 31, &rows[0], &rows[1]);
  to_curve<2>(rows, curve, orient, s_curve, s_rows);
  const uint32_t T = curve[0];
  uint32_t I = curve[1];
  // runs that hold a touched cell, level by level
  const uint32_t t1 = any4(T), t2 = any16(t1), t3 = any_lanes(t2, 2), t4 = any_lanes(t3, 8);
  // the interior cells by the level of their record (the largest untouched run)
  uint32_t c0 = I & t1, c1 = I & ~t1 & t2, c2 = I & ~t2 & t3, c3 = I & ~t3 & t4, c4 = I & ~t4;
  uint32_t tk = T, f1 = t1;
  if (R.geo >> 10) {
    // viewport clip: a record stays when its cell holds lattice points of it
    const CoverQuery Q = A.qs[R.query];
    const int64_t side = (int64_t)1 << sh, y = R.py + lane * side;
    uint32_t row[1] = {0}, box[1];
    if (y < (int64_t)Q.y1 && y + side > (int64_t)Q.y0) {
      // columns with px + m side < x1 and px + (m + 1) side > x0
      const int64_t lo = ((int64_t)Q.x0 - R.px) >> sh, hi = ((int64_t)Q.x1 - 1 - R.px) >> sh;
      if (hi >= 0 && lo <= 31)
        row[0] = (FULL << (lo < 0 ? 0 : lo)) & (FULL >> (31 - (hi > 31 ? 31 : hi)));
    }
    to_curve<1>(row, box, orient, s_curve, s_rows);
    const uint32_t b1 = any4(box[0]), b2 = any16(b1), b3 = any_lanes(b2, 2),
                   b4 = any_lanes(b3, 8);
    tk &= box[0];
    c0 &= box[0];
    c1 &= b1;
    c2 &= b2;
    c3 &= b3;
    c4 &= b4;
    f1 &= b1;
    I = c0 | c1 | c2 | c3 | c4;
  }
  const uint32_t cover = tk | I;
  A.bits[(uint64_t)R.bits * 32 + lane] = cover;
  if (A.flags) A.bbits[(uint64_t)R.bits * 32 + lane] = tk;
  // records in 256ths: a cell of a run of 4^l cells is 1 / 4^l of a record
  S.cells += 256 * (uint32_t)__popc(tk | c0) + 64 * (uint32_t)__popc(c1) +
             16 * (uint32_t)__popc(c2) + 4 * (uint32_t)__popc(c3) + (uint32_t)__popc(c4);
  S.front += __popc(f1 & 0x11111111u);
  S.u[0] |= tk | c0;
  S.u[1] |= c1;
  S.u[2] |= c2;
  S.u[3] |= c3;
  S.u[4] |= c4;
  // positions where this polygon's part of the set changes
  uint32_t prev = __shfl_up_sync(FULL, cover, 1);
  S.starts |= cover ^ ((cover << 1) | (prev >> 31));
  if (A.flags) {
    prev = __shfl_up_sync(FULL, tk, 1);
    S.starts |= tk ^ ((tk << 1) | (prev >> 31));
  }
  const uint32_t last = __shfl_sync(FULL, cover, 31) >> 31;
  const uint32_t blast = A.flags ? __shfl_sync(FULL, tk, 31) >> 31 : 0u;
  if (lane == 0)
    A.info[i] = R.slot | ((cover & 1u) << INFO_FIRST) |
                (A.flags ? (tk & 1u) << (INFO_FIRST + 1) : 0u) | (last << INFO_LAST) |
                (blast << (INFO_LAST + 1)) | INFO_TILE;
}

// two polygons' records that share cells must be the same cell
__device__ __forceinline__ bool records_clash(const uint32_t (&u)[5]) {
  return (u[0] & (u[1] | u[2] | u[3] | u[4])) || (u[1] & (u[2] | u[3] | u[4])) ||
         (u[2] & (u[3] | u[4])) || (u[3] & u[4]);
}

// One warp per tile: the bitmaps of its polygons, what they add to the covering.
// Bound by instruction issue and, a tile being a chain of dependent loads, by the
// warps in flight: with a 64-bit division per edge, a bit-by-bit curve order and
// 92 registers (two blocks per SM) it took 3.06 ms for the 263-zone sweep, with
// small quotients, 2 x 2 blocks and 64 registers 1.26 ms.
__global__ __launch_bounds__(TPB, 4) void tile_raster_kernel(TileArgs A) {
  __shared__ CurveTables s_curve;
  __shared__ __align__(16) uint32_t s_rows[WPB][2][32];
  fill_curve(s_curve);
  __syncthreads();
  if (A.flag[1]) return;  // a crowded tile: the refinement takes over
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t nh = A.heads.n[0];
  for (uint32_t g = blockIdx.x * WPB + w; g < nh; g += gridDim.x * WPB) {
    const uint2 head = A.heads.at[g];
    const uint32_t a = head.x, k = head.y;
    TileSum S;
    for (uint32_t i = a; i < a + k; ++i) raster_element(A, i, lane, s_curve, s_rows[w], S);
    const bool clash = k > 1 && records_clash(S.u);
    if (__any_sync(FULL, clash) && lane == 0) A.flag[2] = 1u;
    if (lane == 0) S.starts &= ~1u;  // the tile's first position is the group's head
    // list entries of the inner starts
    uint32_t ent = 0;
    for (uint32_t i = a; i < a + k; ++i)
      ent += __popc(S.starts & A.bits[(uint64_t)A.rec[i].bits * 32 + lane]);
    const uint32_t ns = __reduce_add_sync(FULL, __popc(S.starts));
    ent = __reduce_add_sync(FULL, ent);
    const uint32_t ncell = __reduce_add_sync(FULL, S.cells);
    const uint32_t fr = __reduce_add_sync(FULL, S.front);
    if (lane == 0) {
      A.inner[a] = ((uint64_t)ns << 32) | ent;
      A.cells[a] = ncell >> 8;
      // frontier size, as the refinement would meet it; spread over counters
      atomicAdd(A.front + (g & (FRONT_SPREAD - 1)), (unsigned long long)fr);
    }
  }
}

// The same by one block per tile, its warps sharing the tile's polygons: a warp takes
// 2.3 us per polygon.
__global__ __launch_bounds__(TPB) void crowd_raster_kernel(TileArgs A) {
  __shared__ CurveTables s_curve;
  __shared__ __align__(16) uint32_t s_rows[WPB][2][32];
  __shared__ uint32_t s_or[6][32];  // starts, u
  __shared__ uint32_t s_sum[3];     // cells, front, entries
  const uint32_t nh = A.heads.n[1];
  if (blockIdx.x >= nh || A.flag[1]) return;
  fill_curve(s_curve);
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (uint32_t g = blockIdx.x; g < nh; g += gridDim.x) {
    const uint2 head = A.heads[A.heads.n[0] + g];
    const uint32_t a = head.x, k = head.y;
    __syncthreads();
    if (threadIdx.x < 6 * 32) s_or[threadIdx.x >> 5][lane] = 0;
    if (threadIdx.x < 3) s_sum[threadIdx.x] = 0;
    __syncthreads();
    TileSum S;
    for (uint32_t i = a + w; i < a + k; i += WPB) raster_element(A, i, lane, s_curve, s_rows[w], S);
    atomicOr(&s_or[0][lane], S.starts);
#pragma unroll
    for (int l = 0; l < 5; ++l) atomicOr(&s_or[1 + l][lane], S.u[l]);
    const uint32_t ncell = __reduce_add_sync(FULL, S.cells);
    const uint32_t fr = __reduce_add_sync(FULL, S.front);
    if (lane == 0) {
      atomicAdd(&s_sum[0], ncell);
      atomicAdd(&s_sum[1], fr);
    }
    __syncthreads();
    uint32_t starts = s_or[0][lane], ent = 0;
    if (lane == 0) starts &= ~1u;
    for (uint32_t i = a + w; i < a + k; i += WPB)
      ent += __popc(starts & A.bits[(uint64_t)A.rec[i].bits * 32 + lane]);
    ent = __reduce_add_sync(FULL, ent);
    if (lane == 0) atomicAdd(&s_sum[2], ent);
    __syncthreads();
    if (w == 0) {
      uint32_t u[5];
#pragma unroll
      for (int l = 0; l < 5; ++l) u[l] = s_or[1 + l][lane];
      const uint32_t ns = __reduce_add_sync(FULL, __popc(starts));
      if (__any_sync(FULL, records_clash(u)) && lane == 0) A.flag[2] = 1u;
      if (lane == 0) {
        A.inner[a] = ((uint64_t)ns << 32) | s_sum[2];
        A.cells[a] = s_sum[0] >> 8;
        atomicAdd(A.front + (g & (FRONT_SPREAD - 1)), (unsigned long long)s_sum[1]);
      }
    }
  }
}

// ---------------------------------------------------------------- elements
// keys of the tile items, appended to the coarse records' keys
__global__ void tile_keys_kernel(const Item* __restrict__ items, uint64_t n,
                                 const uint32_t* __restrict__ pair_query, uint32_t qshift,
                                 uint64_t n_rec, uint64_t* __restrict__ key) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Item it = items[i];
  const uint64_t q = qshift >= 64 ? 0ull : (uint64_t)pair_query[it.pair] << qshift;
  key[n_rec + i] = q | (it.hid << (2 * TILE_DEPTH));
}

__global__ void iota_kernel(uint32_t* __restrict__ p, uint64_t n) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = (uint32_t)i;
}

// The coarse records' info, level and record count, and the tile groups with their
// polygons' records ascending by slot: a tile's element finds its group around it and
// its place among the group's slots.  (One thread inserting a group's records by slot
// took 0.3 ms at 64 polygons, 13 at 500.)
__global__ void element_kernel(const uint64_t* __restrict__ key, const uint32_t* __restrict__ idx,
                               const uint32_t* __restrict__ val, uint64_t n_rec, uint64_t ne,
                               const Item* __restrict__ items,
                               const uint32_t* __restrict__ pair_query,
                               const uint32_t* __restrict__ pair_slot,
                               const CoverQuery* __restrict__ qs, uint32_t B, TileHeads heads,
                               uint32_t* __restrict__ info, uint8_t* __restrict__ level,
                               uint32_t* __restrict__ cells, TileRec* __restrict__ rec,
                               unsigned int* __restrict__ flag) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t k = 0;  // polygons of the group that this element heads
  if (i < ne) {
    const uint32_t el = idx[i];
    if (el < n_rec) {
      const uint32_t v = val[el];
      info[i] = (v & INFO_SLOT) | (1u << INFO_FIRST) | (1u << INFO_LAST);
      level[i] = (uint8_t)((v >> 26) & 31u);
      cells[i] = 1;
    } else {
      level[i] = (uint8_t)TILE_DEPTH;
      info[i] = INFO_TILE;
      // (the sort is stable: a key's coarse cells come before its tiles)
      const uint64_t q = key[i];
      uint64_t a = i, e = i + 1;
      while (a > 0 && i - a < TILE_MAX_GROUP && key[a - 1] == q && idx[a - 1] >= n_rec) --a;
      while (e < ne && e - a <= TILE_MAX_GROUP && key[e] == q) ++e;
      const bool head = a == i;
      if (!head) cells[i] = 0;  // the head's warp counts for the tile
      if (head && i > 0 && key[i - 1] == q) flag[0] = 1u;  // another polygon's cell with the tile's start
      if (e - a > TILE_MAX_GROUP) {
        flag[1] = 1u;
      } else {
        const uint32_t ti = el - (uint32_t)n_rec;
        const Item it = items[ti];
        const uint32_t qi = pair_query[it.pair];
        const CoverQuery Q = qs[qi];
        const uint32_t sh = B - Q.F;
        TileRec R;
        R.px = (int32_t)(it.cx << (sh + TILE_DEPTH));
        R.py = (int32_t)(it.cy << (sh + TILE_DEPTH));
        R.eoff = it.eoff;
        R.ecnt_par = it.ecnt_par;
        R.slot = pair_slot[it.pair];
        const int64_t side = (int64_t)1 << (sh + TILE_DEPTH);
        const bool clip = R.px < (int64_t)Q.x0 || R.py < (int64_t)Q.y0 ||
                          R.px + side > (int64_t)Q.x1 || R.py + side > (int64_t)Q.y1;
        R.geo = sh | (it.orient << 8) | ((uint32_t)clip << 10);
        R.query = qi;
        R.bits = ti;
        uint64_t at = a;
        if (e - a > 1)
#pragma unroll 4
          for (uint64_t j = a; j < e; ++j) {
            const uint32_t o = pair_slot[items[idx[j] - (uint32_t)n_rec].pair];
            at += o < R.slot || (o == R.slot && j < i);
          }
        rec[at] = R;
        if (head) k = (uint32_t)(e - a);
      }
    }
  }
  const uint32_t lane = threadIdx.x & 31;
#pragma unroll
  for (int large = 0; large < 2; ++large) {
    const bool mine = k > 0 && (k > CROWD) == (large != 0);
    const uint32_t b = __ballot_sync(FULL, mine);
    if (!b) continue;
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(heads.n + large, (uint32_t)__popc(b));
    at = __shfl_sync(FULL, at, 0) + __popc(b & ((1u << lane) - 1u));
    if (mine) heads.at[large ? heads.cap - 1 - at : at] = make_uint2((uint32_t)i, k);
  }
}

// ---------------------------------------------------------------- ranges
struct GroupArgs {
  const uint64_t* key;
  const uint32_t* info;
  const uint8_t* level;
  const uint64_t* inner;
  uint64_t ne, lomask;
  uint32_t qshift;
  const CoverQuery* qs;
  // elementary intervals of nested cells (see nested_groups) instead of cells: their
  // ends; inner then holds for every head
  const uint64_t* end;
};

// the first id after element i, whose key is at lo
__device__ __forceinline__ uint64_t end_of(const GroupArgs& A, uint64_t i, uint64_t lo) {
  return A.end ? A.end[i] : lo + (1ull << (2 * A.level[i]));
}
__device__ __forceinline__ uint64_t inner_of(const GroupArgs& A, uint64_t i) {
  return A.end || (A.info[i] & INFO_TILE) ? A.inner[i] : 0ull;
}

__device__ __forceinline__ uint32_t gq(const GroupArgs& A, uint64_t key) {
  return A.qshift >= 64 ? 0u : (uint32_t)(key >> A.qshift);
}
// the list entry of element info at the group's first / last cell
__device__ __forceinline__ uint32_t info_entry(uint32_t v, uint32_t which) {
  return (v & INFO_SLOT) | (((v >> (which + 1)) & 1u) << 31);
}

// A group's entries at its first or last cell, as one ascending list: its elements are
// an ascending run of cells and one of tiles (either may be empty).
struct EndWalk {
  const uint32_t* info;
  uint64_t c, ce, t, te;  // what is left of the runs
  uint32_t which, seen = 0;
  bool ordered = true;
  __device__ EndWalk(const GroupArgs& A, uint64_t a, uint64_t e, uint32_t w)
      : info(A.info), c(a), te(e), which(w) {
    for (ce = a; ce < e && !(info[ce] & INFO_TILE);) ++ce;
    t = ce;
  }
  __device__ uint32_t next() {  // NONE: at the end
    while (c < ce && !((info[c] >> which) & 1u)) ++c;
    while (t < te && !((info[t] >> which) & 1u)) ++t;
    if (c == ce && t == te) return NONE;
    const bool cell = t == te || (c < ce && (info[c] & INFO_SLOT) < (info[t] & INFO_SLOT));
    const uint32_t v = info[cell ? c++ : t++];
    ordered &= (v & INFO_SLOT) >= seen;
    seen = v & INFO_SLOT;
    return info_entry(v, which);
  }
};

// a group's set at its last cell equals another's at its first cell
__device__ bool same_ends(const GroupArgs& A, uint64_t pa, uint64_t pe, uint64_t a, uint64_t e) {
  if (pe - pa > 8 && e - a > 8) {  // side by side: 500 polygons against 500 one by one take 10 ms
    EndWalk x(A, pa, pe, INFO_LAST), y(A, a, e, INFO_FIRST);
    bool same = true;
    for (uint32_t u = 0, v = 0; u != NONE || v != NONE;) {
      u = x.next();
      v = y.next();
      same &= u == v;
      if (!same && !(x.ordered && y.ordered)) break;
    }
    if (same || (x.ordered && y.ordered)) return same;
    // coarser cells of one place are in no order
  }
  uint32_t n0 = 0, n1 = 0;
  for (uint64_t i = pa; i < pe; ++i) n0 += (A.info[i] >> INFO_LAST) & 1u;
  for (uint64_t i = a; i < e; ++i) n1 += (A.info[i] >> INFO_FIRST) & 1u;
  if (n0 != n1) return false;
  for (uint64_t i = a; i < e; ++i) {
    const uint32_t v = A.info[i];
    if (!((v >> INFO_FIRST) & 1u)) continue;
    bool found = false;
    for (uint64_t j = pa; j < pe && !found; ++j)
      found = ((A.info[j] >> INFO_LAST) & 1u) &&
              info_entry(A.info[j], INFO_LAST) == info_entry(v, INFO_FIRST);
    if (!found) return false;
  }
  return true;
}

// Sums over the groups, apart from the packed words (ranges << 32 | list entries) that
// the scan adds up: those carry once there are 2^32 list entries, more than there are
// cells where polygons overlap.  SPREAD counters of ranges, then as many of entries.
struct GroupTotals {
  uint64_t ranges = 0, entries = 0;
};

// Per element: 0, or at the head of a group the ranges it opens (<< 32) and their
// list entries; code: bit 0 an empty gap before it, bit 1 itself, bit 2 the empty
// tail of its query, bit 3 the query's first group, bit 4 its last.  A gap, a
// group or a tail opens a range when its set differs from what comes before.
__device__ uint64_t count_group(const GroupArgs& A, uint64_t a, uint8_t* __restrict__ code,
                                uint32_t* __restrict__ qhead, unsigned int* __restrict__ flag) {
  const uint64_t key = A.key[a];
  if (a > 0 && A.key[a - 1] == key) {
    code[a] = 0;
    return 0;
  }
  const uint32_t q = gq(A, key);
  const uint64_t lo = key & A.lomask, hi = end_of(A, a, lo);
  bool nest = false;
  uint32_t nfirst = 0, nlast = 0;
  uint64_t e = a;
  for (; e < A.ne && A.key[e] == key; ++e) {
    const uint32_t v = A.info[e];
    if (!A.end) nest |= A.level[e] != A.level[a] || ((v ^ A.info[a]) & INFO_TILE);
    nfirst += (v >> INFO_FIRST) & 1u;
    nlast += (v >> INFO_LAST) & 1u;
  }
  const bool first = a == 0 || gq(A, A.key[a - 1]) != q;
  const bool last = e == A.ne || gq(A, A.key[e]) != q;
  bool gap = lo > 0, opens_gap = gap, opens_head = gap ? nfirst != 0 : true;
  if (!first) {
    const uint64_t pkey = A.key[a - 1];
    uint64_t pa = a - 1;
    bool plast = (A.info[pa] >> INFO_LAST) & 1u;
    while (pa > 0 && A.key[pa - 1] == pkey) {
      --pa;
      plast |= (A.info[pa] >> INFO_LAST) & 1u;
    }
    const uint64_t pend = end_of(A, pa, pkey & A.lomask);
    nest |= lo < pend;  // the previous cell reaches into this one
    gap = lo > pend;
    opens_gap = gap && plast;
    opens_head = gap ? nfirst != 0 : !same_ends(A, pa, a, a, e);
  }
  const bool opens_tail = last && hi < (1ull << (2 * A.qs[q].F)) && nlast != 0;
  code[a] = (uint8_t)(opens_gap | (opens_head << 1) | (opens_tail << 2) | (first << 3) | (last << 4));
  if (first) qhead[q] = (uint32_t)a;
  if (nest) flag[0] = 1u;
  // one group's entries fit: a tile's 1024 positions times TILE_MAX_GROUP + MAX_OVERLAP
  return inner_of(A, a) + ((uint64_t)(opens_gap + opens_head + opens_tail) << 32) +
         (opens_head ? nfirst : 0u);
}

__global__ __launch_bounds__(256) void group_count_kernel(GroupArgs A, uint64_t* __restrict__ cnt,
                                                          uint8_t* __restrict__ code,
                                                          uint32_t* __restrict__ qhead,
                                                          unsigned int* __restrict__ flag,
                                                          unsigned long long* __restrict__ sums) {
  __shared__ uint32_t s_sum[2][8];
  if (flag[1]) return;  // (a crowded tile: nothing is made)
  const uint64_t a = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  uint64_t c = 0;
  if (a < A.ne) cnt[a] = c = count_group(A, a, code, qhead, flag);
  const uint32_t r = __reduce_add_sync(FULL, (uint32_t)(c >> 32));
  const uint32_t l = __reduce_add_sync(FULL, (uint32_t)c);
  if ((threadIdx.x & 31) == 0) {
    s_sum[0][threadIdx.x >> 5] = r;
    s_sum[1][threadIdx.x >> 5] = l;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    unsigned long long t = 0;
    for (int w = 0; w < 8; ++w) t += s_sum[threadIdx.x][w];
    if (t) atomicAdd(sums + threadIdx.x * SPREAD + (blockIdx.x & (SPREAD - 1)), t);
  }
}

struct RangeOut {
  const QueryOut* q;
  uint64_t* qopen;  // per query: ranges before its first group, after its last
  uint32_t* qlist;  // per query: list entries before its first group, after its last
};

// inserts v into the list out[0, t) by slot, which ascends up to *last, its last entry
__device__ __forceinline__ void insert_entry(uint32_t* out, uint32_t t, uint32_t v, uint32_t* last) {
  uint32_t j = t;
  if (t > 0 && (*last & INFO_SLOT) > (v & INFO_SLOT)) {
    while (j > 0 && (out[j - 1] & INFO_SLOT) > (v & INFO_SLOT)) {
      out[j] = out[j - 1];
      --j;
    }
  } else {
    *last = v;
  }
  out[j] = v;
}

// the ranges and list entries before each query's first group (~0: no records)
__global__ void query_offsets_kernel(const uint32_t* __restrict__ qhead, uint32_t Q,
                                     const uint64_t* __restrict__ off, uint64_t* __restrict__ qoff) {
  const uint32_t q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < Q) qoff[q] = qhead[q] == NONE ? ~0ull : off[qhead[q]];
}

__device__ __forceinline__ uint32_t pay_of(uint32_t n, uint32_t entry, uint64_t e) {
  return n == 0 ? NONE
         : n == 1 ? (entry & INFO_SLOT) | ((entry >> 31) << 30)
                  : 0x80000000u | (uint32_t)e;
}

// the ranges outside the tiles: gaps, groups' first ranges, tails
__global__ void group_emit_kernel(GroupArgs A, const uint64_t* __restrict__ off,
                                  const uint8_t* __restrict__ code,
                                  const uint64_t* __restrict__ extra, RangeOut o) {
  const uint64_t a = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= A.ne) return;
  const uint64_t key = A.key[a];
  if (a > 0 && A.key[a - 1] == key) return;
  const uint32_t c = code[a], q = gq(A, key);
  const uint64_t lo = key & A.lomask, hi = end_of(A, a, lo);
  uint64_t ro = off[a] >> 32;
  uint32_t L = (uint32_t)off[a];
  if (c & 8u) {
    o.qopen[2 * q] = ro;
    o.qlist[2 * q] = L;
  }
  uint64_t e = ro + extra[q];
  const QueryOut O = o.q[q];
  if (c & 1u) {
    uint64_t from = 0;
    if (!(c & 8u)) {  // the end of the previous group's cell
      const uint64_t pkey = A.key[a - 1];
      from = end_of(A, a - 1, pkey & A.lomask);
    }
    O.start[e] = from;
    O.list_off[e] = L - O.l0;
    O.pay[e] = NONE;
    ++e;
  }
  if (c & 2u) {
    uint32_t n = 0, one = 0, top = 0;
    for (uint64_t i = a; i < A.ne && A.key[i] == key; ++i) {
      const uint32_t v = A.info[i];
      if (!((v >> INFO_FIRST) & 1u)) continue;
      one = info_entry(v, INFO_FIRST);
      insert_entry(O.list_ids + L, n++, one, &top);
    }
    O.start[e] = lo;
    O.list_off[e] = L - O.l0;
    O.pay[e] = pay_of(n, one, e - O.e0);
    L += n;
    ++e;
  }
  const uint64_t in = inner_of(A, a);
  e += in >> 32;
  L += (uint32_t)in;
  if (c & 4u) {
    O.start[e] = hi;
    O.list_off[e] = L - O.l0;
    O.pay[e] = NONE;
    ++e;
  }
  if (c & 16u) {
    o.qopen[2 * q + 1] = e - extra[q];
    o.qlist[2 * q + 1] = L;
  }
}

// The ranges that start inside a tile, one warp per tile.  The start positions are
// listed in shared memory first, so that lane i then makes the i-th of 32 ranges
// and the arrays are written side by side.  A tile is a chain of dependent reads;
// a warp takes up to 32 tiles in a row, its lanes read what belongs to one tile each
// at once, and a tile's polygon records are read while the tile before is written.
// (263-zone sweep: 1.02 ms with each lane making the ranges of its own positions,
// 0.67 with the list, 0.61 with the reads ahead; 0.79 before them with a sweep's
// own arrays per covering.)
// BASE: polygons whose coarser cells hold the whole tile come on top (base: per tile
// its group's first element, of which the base polygons are the first ones).
struct TileBase {
  const uint2* at;       // per tile head: its group's first element, base polygons
  const uint32_t* info;  // the groups' elements
};
template <bool BASE>
__global__ __launch_bounds__(TPB) void tile_emit_kernel(TileArgs A, const uint64_t* __restrict__ off,
                                                        const uint8_t* __restrict__ code,
                                                        const uint64_t* __restrict__ extra,
                                                        uint64_t lomask, TileBase base,
                                                        RangeOut o) {
  constexpr uint32_t STAGE = 4;  // polygons of a tile held in registers and shared memory
  __shared__ uint32_t s_h[WPB][STAGE][32];
  __shared__ uint16_t s_pos[WPB][1024];
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t nh = A.heads.n[0];
  // tiles in a row per warp: 32, fewer when there are not enough for all warps
  const uint32_t run = min(32u, max(1u, nh / (gridDim.x * WPB)));
  for (uint32_t g0 = (blockIdx.x * WPB + w) * run; g0 < nh; g0 += gridDim.x * WPB * run) {
   const uint32_t in_run = min(run, nh - g0);
   uint2 my_head = make_uint2(0, 0);
   uint64_t my_key = 0, my_pre = 0;
   uint32_t my_ns = 0, my_c = 0;
   uint2 my_base = make_uint2(0, 0);
   if (lane < in_run) {
     my_head = A.heads.at[g0 + lane];
     my_base = BASE ? base.at[my_head.x] : make_uint2(my_head.x, 0);
     my_ns = (uint32_t)(A.inner[my_head.x] >> 32);
     my_key = A.key[my_head.x];
     my_pre = off[my_base.x];
     my_c = code[my_base.x];
   }
   uint32_t nb = 0, nslot = 0;  // lane j: polygon j's bitmap and slot, of the next tile
   auto fetch = [&](uint32_t i) {
     const uint32_t ia = __shfl_sync(FULL, my_head.x, i), ik = __shfl_sync(FULL, my_head.y, i);
     if (lane < ik) {
       nb = A.rec[ia + lane].bits;
       nslot = A.rec[ia + lane].slot;
     }
   };
   fetch(0);
   for (uint32_t i = 0; i < in_run; ++i) {
    const uint32_t a = __shfl_sync(FULL, my_head.x, i), k = __shfl_sync(FULL, my_head.y, i);
    const uint32_t ns = __shfl_sync(FULL, my_ns, i), c = __shfl_sync(FULL, my_c, i);
    const uint64_t key = __shfl_sync(FULL, (unsigned long long)my_key, i);
    const uint64_t pre = __shfl_sync(FULL, (unsigned long long)my_pre, i);
    const uint32_t rb = nb, rslot = nslot;
    uint32_t h[STAGE];
#pragma unroll
    for (uint32_t j = 0; j < STAGE; ++j) {
      const uint32_t at = __shfl_sync(FULL, rb, j);
      h[j] = j < k && ns ? A.bits[(uint64_t)at * 32 + lane] : 0u;
    }
    if (i + 1 < in_run) fetch(i + 1);
    if (ns == 0) continue;
    uint32_t starts = 0, nfirst = 0;
    auto changes = [&](uint32_t v) {
      const uint32_t prev = __shfl_up_sync(FULL, v, 1);
      starts |= v ^ ((v << 1) | (prev >> 31));
    };
    __syncwarp();
#pragma unroll
    for (uint32_t j = 0; j < STAGE; ++j) {
      changes(h[j]);
      nfirst += __shfl_sync(FULL, h[j], 0) & 1u;
      s_h[w][j][lane] = h[j];
    }
    for (uint32_t j = STAGE; j < k; ++j) {
      const uint32_t v = A.bits[(uint64_t)A.rec[a + j].bits * 32 + lane];
      changes(v);
      nfirst += __shfl_sync(FULL, v, 0) & 1u;
    }
    if (A.flags)
      for (uint32_t j = 0; j < k; ++j) changes(A.bbits[(uint64_t)A.rec[a + j].bits * 32 + lane]);
    if (lane == 0) starts &= ~1u;
    uint32_t at = __popc(starts);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t t = __shfl_up_sync(FULL, at, d);
      if (lane >= (uint32_t)d) at += t;
    }
    at -= __popc(starts);
    for (uint32_t m = starts; m; m &= m - 1) s_pos[w][at++] = (uint16_t)(32 * lane + __ffs(m) - 1);
    __syncwarp();
    const uint32_t q = A.qshift >= 64 ? 0u : (uint32_t)(key >> A.qshift);
    uint64_t e0 = (pre >> 32) + extra[q] + (c & 1u) + ((c >> 1) & 1u);
    const uint32_t b0 = BASE ? __shfl_sync(FULL, my_base.x, i) : 0u;
    const uint32_t nb0 = BASE ? __shfl_sync(FULL, my_base.y, i) : 0u;
    uint32_t L0 = (uint32_t)pre + ((c & 2u) ? nfirst + nb0 : 0u);
    const uint64_t lo = key & lomask;
    const QueryOut O = o.q[q];
    uint32_t slots[STAGE];
#pragma unroll
    for (uint32_t j = 0; j < STAGE; ++j) slots[j] = __shfl_sync(FULL, rslot, j);
    for (uint32_t i0 = 0; i0 < ns; i0 += 32) {
      const bool on = i0 + lane < ns;
      const uint32_t pos = on ? s_pos[w][i0 + lane] : 0u;
      const uint32_t wi = pos >> 5, bi = pos & 31u;
      // the polygons of the range: bit j of set for the staged ones
      uint32_t set = 0;
#pragma unroll
      for (uint32_t j = 0; j < STAGE; ++j) set |= ((s_h[w][j][wi] >> bi) & 1u) << j;
      if (!on) set = 0;
      uint32_t n = __popc(set);
      auto more = [&](uint32_t j) {
        return (A.bits[(uint64_t)A.rec[a + j].bits * 32 + wi] >> bi) & 1u;
      };
      if (on)
        for (uint32_t j = STAGE; j < k; ++j) n += more(j);
      if (BASE && on) n += nb0;
      uint32_t inc = n;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL, inc, d);
        if (lane >= (uint32_t)d) inc += t;
      }
      if (on) {
        const uint64_t e = e0 + i0 + lane;
        const uint32_t L = L0 + inc - n;
        uint32_t one = 0, t = L;
        uint32_t bi0 = 0;  // base polygons written (they ascend too)
        auto put_base = [&](uint32_t below) {
          for (; (int)bi0 < (int)nb0; ++bi0) {
            const uint32_t v = base.info[b0 + bi0] & INFO_SLOT;
            if (v >= below) break;
            one = v;
            O.list_ids[t++] = v;
          }
        };
        auto put = [&](uint32_t j, uint32_t slot) {  // the polygons ascend by slot
          put_base(slot);
          one = slot;
          if (A.flags) one |= ((A.bbits[(uint64_t)A.rec[a + j].bits * 32 + wi] >> bi) & 1u) << 31;
          O.list_ids[t++] = one;
        };
#pragma unroll
        for (uint32_t j = 0; j < STAGE; ++j)
          if ((set >> j) & 1u) put(j, slots[j]);
        for (uint32_t j = STAGE; j < k; ++j)
          if (more(j)) put(j, A.rec[a + j].slot);
        put_base(~0u);
        O.start[e] = lo + pos;
        O.list_off[e] = L - O.l0;
        O.pay[e] = pay_of(n, one, e - O.e0);
      }
      L0 += __shfl_sync(FULL, inc, 31);
    }
   }
  }
}

// The same by one block per tile of more than CROWD polygons, its warps sharing first
// the polygons, then the ranges, 32 at a time against 32 polygons with several reads in
// flight.  (512 polygons over one another, 32 x 32 tiles of them: the build 15.5 ms with
// a warp per tile and one thread ordering its polygons, 6.5 ms; 500 small polygons in one
// tile 16 -> 0.8 ms.)
template <bool BASE>
__global__ __launch_bounds__(TPB) void crowd_emit_kernel(TileArgs A, const uint64_t* __restrict__ off,
                                                         const uint8_t* __restrict__ code,
                                                         const uint64_t* __restrict__ extra,
                                                         uint64_t lomask, TileBase base,
                                                         RangeOut o) {
  __shared__ uint32_t s_starts[32], s_first;
  __shared__ uint16_t s_pos[1024];
  __shared__ uint32_t s_list[1024];  // the ranges' list entries, then what is before them
  const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t nh = A.heads.n[1];
  for (uint32_t g = blockIdx.x; g < nh; g += gridDim.x) {
    const uint2 head = A.heads[A.heads.n[0] + g];
    const uint32_t a = head.x, k = head.y;
    const uint32_t ns = (uint32_t)(A.inner[a] >> 32);
    if (ns == 0) continue;  // the whole block
    const uint2 hb = BASE ? base.at[a] : make_uint2(a, 0);
    const uint32_t nb0 = hb.y;  // base polygons
    const uint64_t key = A.key[a], pre = off[hb.x], lo = key & lomask;
    const uint32_t c = code[hb.x];
    const uint32_t q = A.qshift >= 64 ? 0u : (uint32_t)(key >> A.qshift);
    const QueryOut O = o.q[q];
    __syncthreads();
    if (threadIdx.x < 32) s_starts[lane] = 0;
    if (threadIdx.x == 0) s_first = 0;
    __syncthreads();
    uint32_t starts = 0, first = 0;
    auto changes = [&](uint32_t v) {
      const uint32_t prev = __shfl_up_sync(FULL, v, 1);
      starts |= v ^ ((v << 1) | (prev >> 31));
    };
    for (uint32_t i = a + w; i < a + k; i += WPB) {
      const uint64_t at = (uint64_t)A.rec[i].bits * 32 + lane;
      const uint32_t v = A.bits[at];
      first += v & 1u;  // (lane 0's is the tile's first position)
      changes(v);
      if (A.flags) changes(A.bbits[at]);
    }
    atomicOr(&s_starts[lane], starts);
    if (lane == 0) atomicAdd(&s_first, first);
    __syncthreads();
    if (w == 0) {
      starts = lane == 0 ? s_starts[0] & ~1u : s_starts[lane];
      uint32_t at = __popc(starts);
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t t = __shfl_up_sync(FULL, at, d);
        if (lane >= (uint32_t)d) at += t;
      }
      at -= __popc(starts);
      for (uint32_t m = starts; m; m &= m - 1) s_pos[at++] = (uint16_t)(32 * lane + __ffs(m) - 1);
    }
    __syncthreads();
    // bit j: polygon j0 + j holds the position (all lanes take part)
    auto members = [&](uint32_t j0, uint32_t pos, bool on) {
      const uint32_t m = min(32u, k - j0), id = lane < m ? A.rec[a + j0 + lane].bits : 0u;
      uint32_t v = 0;
#pragma unroll 8
      for (uint32_t j = 0; j < m; ++j)
        v |= ((A.bits[(uint64_t)__shfl_sync(FULL, id, j) * 32 + (pos >> 5)] >> (pos & 31u)) & 1u) << j;
      return on ? v : 0u;
    };
    for (uint32_t i0 = w * 32; i0 < ns; i0 += TPB) {
      const bool on = i0 + lane < ns;
      const uint32_t pos = on ? s_pos[i0 + lane] : 0u;
      uint32_t n = nb0;
      for (uint32_t j0 = 0; j0 < k; j0 += 32) n += __popc(members(j0, pos, on));
      if (on) s_list[i0 + lane] = n;
    }
    __syncthreads();
    if (w == 0) {
      uint32_t sum = 0;
      for (uint32_t i0 = 0; i0 < ns; i0 += 32) {
        const uint32_t n = i0 + lane < ns ? s_list[i0 + lane] : 0u;
        uint32_t inc = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t t = __shfl_up_sync(FULL, inc, d);
          if (lane >= (uint32_t)d) inc += t;
        }
        if (i0 + lane < ns) s_list[i0 + lane] = sum + inc - n;
        sum += __shfl_sync(FULL, inc, 31);
      }
    }
    __syncthreads();
    const uint64_t e0 = (pre >> 32) + extra[q] + (c & 1u) + ((c >> 1) & 1u);
    const uint32_t L0 = (uint32_t)pre + ((c & 2u) ? s_first + nb0 : 0u);
    for (uint32_t i0 = w * 32; i0 < ns; i0 += TPB) {
      const bool on = i0 + lane < ns;
      const uint32_t pos = on ? s_pos[i0 + lane] : 0u;
      const uint32_t L = on ? L0 + s_list[i0 + lane] : 0u;
      uint32_t one = 0, t = L, b = 0;  // b: base polygons written (they ascend too)
      auto put_base = [&](uint32_t below) {
        for (; b < nb0; ++b) {
          const uint32_t v = base.info[hb.x + b] & INFO_SLOT;
          if (v >= below) break;
          O.list_ids[t++] = one = v;
        }
      };
      for (uint32_t j0 = 0; j0 < k; j0 += 32)
        for (uint32_t m = members(j0, pos, on); m; m &= m - 1) {
          const TileRec& R = A.rec[a + j0 + __ffs(m) - 1];
          const uint32_t slot = R.slot;
          if (BASE) put_base(slot);
          one = slot;
          if (A.flags)
            one |= ((A.bbits[(uint64_t)R.bits * 32 + (pos >> 5)] >> (pos & 31u)) & 1u) << 31;
          O.list_ids[t++] = one;
        }
      if (on) {
        if (BASE) put_base(~0u);
        const uint64_t e = e0 + i0 + lane;
        O.start[e] = lo + pos;
        O.list_off[e] = L - O.l0;
        O.pay[e] = pay_of(t - L, one, e - O.e0);
      }
    }
  }
}

// ---------------------------------------------------------------- nested cells
// One query whose polygons overlap: a coarser cell of one polygon may hold cells and
// tiles of others.  The elements' ends cut the ids into elementary intervals, each a
// tile or free of them; a coarser cell counts for every interval it spans.  The
// intervals' polygons (in slot order), then their tiles', become the elements of
// groups like the ones above, an interval each.  Only the few coarse cells are
// sorted and paired, where the refinement to the finest level does so with every
// cell: 64 stars with holes at eps 64, uploaded, covered, indexed and joined, 1600 us
// -> 1069 us.  A group's set is compared and ordered by one thread; polygons laid over
// one another, eps 64 and 16, refinement -> here: 2 of them 0.87 -> 0.60 and 1.06
// -> 0.71 ms, 64: 1.70 -> 0.92 and 4.12 -> 1.32, 512: 29.6 -> 10.8 and 268 -> 26 (before
// blocks shared the tiles of many polygons; 511 on a 2^13 grid now 11.7 -> 4.0 and 139 -> 6.5).
// With more than MAX_OVERLAP over one another the refinement takes over.

__global__ void ends_kernel(const uint64_t* __restrict__ key, const uint8_t* __restrict__ level,
                            uint64_t ne, uint64_t top, uint64_t* __restrict__ bp) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < ne) {
    bp[2 * i] = key[i];
    bp[2 * i + 1] = key[i] + (1ull << (2 * level[i]));
  } else if (i == ne) {
    bp[2 * ne] = 0;
    bp[2 * ne + 1] = top;
  }
}

__device__ __forceinline__ uint32_t place_of(const uint64_t* __restrict__ b, uint32_t m, uint64_t v) {
  uint32_t lo = 0;
  for (uint32_t len = m; len > 0;) {
    const uint32_t half = len >> 1;
    if (b[lo + half] < v) {
      lo += half + 1;
      len -= half + 1;
    } else {
      len = half;
    }
  }
  return lo;
}

// per element its first interval and how many it spans (a tile: none, its own)
__global__ void element_spans_kernel(const uint64_t* __restrict__ key,
                                     const uint8_t* __restrict__ level,
                                     const uint32_t* __restrict__ info, uint64_t ne,
                                     const uint64_t* __restrict__ b, uint32_t m,
                                     uint32_t* __restrict__ first, uint32_t* __restrict__ span) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ne) return;
  const uint32_t k = place_of(b, m, key[i]);
  first[i] = k;
  span[i] = (info[i] & INFO_TILE) ? 0u : place_of(b, m, key[i] + (1ull << (2 * level[i]))) - k;
}

// pair i of (interval, slot): of the element e with poff[e] <= i < poff[e + 1]
__global__ void span_pairs_kernel(const uint64_t* __restrict__ poff, uint64_t ne,
                                  const uint32_t* __restrict__ first,
                                  const uint32_t* __restrict__ info, uint64_t T, uint32_t pbits,
                                  uint64_t* __restrict__ pairs) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= T) return;
  uint64_t e = 0;
  for (uint64_t len = ne; len > 1;) {
    const uint64_t half = len >> 1;
    if (poff[e + half] <= i) e += half;
    len -= half;
  }
  pairs[i] = ((uint64_t)(first[e] + (uint32_t)(i - poff[e])) << pbits) | (info[e] & INFO_SLOT);
}

__global__ void pair_lengths_kernel(const uint64_t* __restrict__ pairs, uint64_t T, uint32_t pbits,
                                    uint32_t* __restrict__ len, uint32_t* __restrict__ count,
                                    unsigned int* __restrict__ flag) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= T) return;
  const uint32_t k = (uint32_t)(pairs[i] >> pbits);
  if (atomicAdd(&len[k], 1u) == MAX_OVERLAP) flag[1] = 1u;
  atomicAdd(&count[k], 1u);
}
__global__ void tile_lengths_kernel(TileHeads heads, const uint32_t* __restrict__ first,
                                    uint32_t* __restrict__ count) {
  const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < heads.all()) atomicAdd(&count[first[heads[g].x]], heads[g].y);
}

struct NestedOut {
  uint64_t* key;
  uint64_t* end;
  uint32_t* info;
  uint64_t* inner;
  uint2* base;  // per tile head (by its old element): group's first element, base polygons
};
__global__ void base_elements_kernel(const uint64_t* __restrict__ pairs, uint64_t T, uint32_t pbits,
                                     const uint64_t* __restrict__ b,
                                     const uint32_t* __restrict__ eoff,
                                     const uint32_t* __restrict__ poff, NestedOut o) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= T) return;
  const uint32_t k = (uint32_t)(pairs[i] >> pbits);
  const uint32_t at = eoff[k] + (uint32_t)(i - poff[k]);
  o.key[at] = b[k];
  o.end[at] = b[k + 1];
  o.info[at] = (uint32_t)(pairs[i] & ((1ull << pbits) - 1)) | (1u << INFO_FIRST) | (1u << INFO_LAST);
}
__global__ void tile_elements_kernel(TileHeads heads, const uint32_t* __restrict__ first,
                                     const uint32_t* __restrict__ info,
                                     const uint64_t* __restrict__ inner,
                                     const uint64_t* __restrict__ b,
                                     const uint32_t* __restrict__ len,
                                     const uint32_t* __restrict__ eoff, NestedOut o) {
  const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= heads.all()) return;
  const uint2 h = heads[g];
  const uint32_t k = first[h.x], e = eoff[k], n = len[k];
  for (uint32_t j = 0; j < h.y; ++j) {
    o.key[e + n + j] = b[k];
    o.end[e + n + j] = b[k + 1];
    o.info[e + n + j] = info[h.x + j];
  }
  // every range that starts inside the tile lists the base polygons too
  const uint64_t in = inner[h.x];
  o.inner[e] = in + (uint64_t)n * (uint32_t)(in >> 32);
  o.base[h.x] = make_uint2(e, n);
}

// the groups of nested cells: *ga, their number of elements *ne2, and the tiles'
// base polygons, all from sc
sdb_status nested_groups(const TileArgs& ta, const uint8_t* level, uint64_t n_tile, uint32_t F,
                         uint32_t slots, Scratch& sc, cudaStream_t s, GroupArgs* ga, TileBase* tb) {
  const uint64_t ne = ta.ne, nbp = 2 * ne + 2, top = 1ull << (2 * F);
  uint64_t *bp, *bptmp, *bps, *b, *poff, *dT;
  uint32_t *first, *span;
  SDB_TRY(sc.get(&bp, nbp));
  SDB_TRY(sc.get(&bptmp, nbp));
  SDB_TRY(sc.get(&b, nbp));
  SDB_TRY(sc.get(&first, ne));
  SDB_TRY(sc.get(&span, ne));
  SDB_TRY(sc.get(&poff, ne));
  SDB_TRY(sc.get(&dT, 1));
  ends_kernel<<<grid_for(ne + 1, 256), 256, 0, s>>>(ta.key, level, ne, top, bp);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  SDB_TRY(radix_sort_keys(bp, bptmp, nbp, 2 * (int)(F - TILE_DEPTH) + 1, s, &bps, 2 * TILE_DEPTH));
  size_t m = 0;
  SDB_TRY(unique_sorted(bps, nbp, b, &m, s));
  if (m < 2 || m > 0xfffffff0ull) {
    set_error("covering: %zu breakpoints out of range", m);
    return SDB_EINVAL;
  }
  const uint32_t nint = (uint32_t)m - 1;
  element_spans_kernel<<<grid_for(ne, 256), 256, 0, s>>>(ta.key, level, ta.info, ne, b, (uint32_t)m,
                                                        first, span);
  note_launch();
  SDB_TRY_CUDA(cudaGetLastError());
  SDB_TRY(exclusive_scan_u32(span, poff, ne, dT, s));
  uint64_t T = 0;
  SDB_TRY_CUDA(cudaMemcpyAsync(&T, dT, 8, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaStreamSynchronize(s));
  if (T + n_tile >= 0xffffffffull) {
    set_error("covering: %llu (interval, polygon) pairs exceed the 32-bit list range",
              (unsigned long long)T);
    return SDB_ENOMEM;
  }
  uint32_t pbits = 1, ibits = 1;
  while (pbits < 32 && (slots - 1) >> pbits) ++pbits;
  while (ibits < 32 && nint >> ibits) ++ibits;
  const uint64_t ne2 = T + n_tile;
  uint64_t *pairs, *ptmp, *ps;
  uint32_t *len, *count, *eoff, *loff;
  NestedOut no{};
  SDB_TRY(sc.get(&pairs, T));
  SDB_TRY(sc.get(&ptmp, T));
  SDB_TRY(sc.get(&len, nint));
  SDB_TRY(sc.get(&count, nint));
  SDB_TRY(sc.get(&eoff, nint));
  SDB_TRY(sc.get(&loff, nint));
  SDB_TRY(sc.get(&no.key, ne2));
  SDB_TRY(sc.get(&no.end, ne2));
  SDB_TRY(sc.get(&no.info, ne2));
  SDB_TRY(sc.get(&no.inner, ne2));
  SDB_TRY(sc.get(&no.base, ne));
  SDB_TRY_CUDA(cudaMemsetAsync(len, 0, (size_t)nint * 4, s));
  SDB_TRY_CUDA(cudaMemsetAsync(count, 0, (size_t)nint * 4, s));
  SDB_TRY_CUDA(cudaMemsetAsync(no.inner, 0, (size_t)ne2 * 8, s));
  ps = pairs;
  if (T) {
    span_pairs_kernel<<<grid_for(T, 256), 256, 0, s>>>(poff, ne, first, ta.info, T, pbits, pairs);
    note_launch();
    SDB_TRY_CUDA(cudaGetLastError());
    SDB_TRY(radix_sort_keys(pairs, ptmp, T, (int)(pbits + ibits), s, &ps));
    pair_lengths_kernel<<<grid_for(T, 256), 256, 0, s>>>(ps, T, pbits, len, count, ta.flag);
    note_launch();
  }
  if (n_tile) {
    tile_lengths_kernel<<<grid_for(n_tile, 256), 256, 0, s>>>(ta.heads, first, count);
    note_launch();
  }
  SDB_TRY_CUDA(cudaGetLastError());
  SDB_TRY(exclusive_scan<uint32_t>(len, loff, nint, nullptr, s));
  SDB_TRY(exclusive_scan<uint32_t>(count, eoff, nint, nullptr, s));
  if (T) {
    base_elements_kernel<<<grid_for(T, 256), 256, 0, s>>>(ps, T, pbits, b, eoff, loff, no);
    note_launch();
  }
  if (n_tile) {
    tile_elements_kernel<<<grid_for(n_tile, 256), 256, 0, s>>>(ta.heads, first, ta.info, ta.inner, b, len,
                                                              eoff, no);
    note_launch();
  }
  SDB_TRY_CUDA(cudaGetLastError());
  ga->key = no.key;
  ga->info = no.info;
  ga->inner = no.inner;
  ga->end = no.end;
  ga->ne = ne2;
  *tb = TileBase{no.base, no.info};
  return SDB_OK;
}

GroupTotals group_totals(const unsigned long long* sums) {
  GroupTotals t;
  for (uint32_t i = 0; i < SPREAD; ++i) {
    t.ranges += sums[i];
    t.entries += sums[SPREAD + i];
  }
  return t;
}

// list offsets are 32-bit numbers (a test builds this file with a smaller limit)
#ifndef SDB_LIST_LIMIT
#define SDB_LIST_LIMIT 0xffffffffull
#endif
constexpr uint64_t LIST_LIMIT = SDB_LIST_LIMIT;

}  // namespace

sdb_status cover_tiles(const uint64_t* rkey, const uint32_t* rval, uint64_t n_rec, const Item* items,
                       uint64_t n_tile, const uint32_t* elist, const Edge* edges,
                       const uint32_t* pair_query, const uint32_t* pair_slot,
                       const CoverQuery* d_qs, const CoverSpec& spec, uint32_t qshift,
                       int key_bits, cudaStream_t s, CoverSet* out, TileOutcome* outcome) {
  TraceScope tr("cover.tiles", s);
  *outcome = TileOutcome::made;
  Scratch sc(s);
  const uint32_t Q = spec.Q;
  const uint64_t ne = n_rec + n_tile;
  if (ne >= 0xffffffffull) {
    set_error("covering: %llu cells exceed the 32-bit index range", (unsigned long long)ne);
    return SDB_ENOMEM;
  }
  uint64_t *keys, *ktmp, *sk;
  uint32_t *ix, *ixtmp, *si;
  SDB_TRY(sc.get(&keys, ne));
  SDB_TRY(sc.get(&ktmp, ne));
  SDB_TRY(sc.get(&ix, ne));
  SDB_TRY(sc.get(&ixtmp, ne));
  if (n_rec)
    SDB_TRY_CUDA(cudaMemcpyAsync(keys, rkey, n_rec * 8, cudaMemcpyDeviceToDevice, s));
  if (n_tile) {
    tile_keys_kernel<<<grid_for(n_tile, 256), 256, 0, s>>>(items, n_tile, pair_query, qshift, n_rec,
                                                          keys);
    note_launch();
  }
  if (ne) {
    iota_kernel<<<grid_for(ne, 256), 256, 0, s>>>(ix, ne);
    note_launch();
  }
  SDB_TRY_CUDA(cudaGetLastError());
  {
    // every element starts on a multiple of a tile: the low key bits are zero
    TraceScope tr1("cover.sort", s);
    SDB_TRY(radix_sort_pairs(keys, ix, ktmp, ixtmp, ne, key_bits - 2 * TILE_DEPTH, s, &sk, &si,
                             nullptr, 2 * TILE_DEPTH));
  }
  uint2* heads;
  TileRec* rec;
  uint32_t *info, *cells, *bits, *bbits = nullptr, *qhead;
  uint8_t *level, *code;
  uint64_t *inner, *cnt, *off, *coff, *tot;
  // nested, crowded, overlapping inside tiles; then the numbers of tile groups
  unsigned int* dflag;
  unsigned long long *front, *sums;  // the last level's frontier, GroupTotals
  SDB_TRY(sc.get(&heads, n_tile));
  SDB_TRY(sc.get(&rec, ne));
  SDB_TRY(sc.get(&info, ne));
  SDB_TRY(sc.get(&cells, ne));
  SDB_TRY(sc.get(&level, ne));
  SDB_TRY(sc.get(&code, ne));
  SDB_TRY(sc.get(&inner, ne));
  SDB_TRY(sc.get(&cnt, ne));
  SDB_TRY(sc.get(&off, ne));
  SDB_TRY(sc.get(&coff, ne));
  SDB_TRY(sc.get(&tot, 2));
  SDB_TRY(sc.get(&qhead, Q));
  SDB_TRY(sc.get(&dflag, 5));
  SDB_TRY(sc.get(&front, FRONT_SPREAD + 2 * SPREAD));
  sums = front + FRONT_SPREAD;
  SDB_TRY(sc.get(&bits, n_tile * 32));
  if (spec.flags) SDB_TRY(sc.get(&bbits, n_tile * 32));
  SDB_TRY_CUDA(cudaMemsetAsync(dflag, 0, 20, s));
  SDB_TRY_CUDA(cudaMemsetAsync(tot, 0, 16, s));
  SDB_TRY_CUDA(cudaMemsetAsync(front, 0, (FRONT_SPREAD + 2 * SPREAD) * 8, s));
  SDB_TRY_CUDA(cudaMemsetAsync(qhead, 0xff, (size_t)Q * 4, s));
  TileArgs ta{};
  ta.rec = rec;
  ta.elist = elist;
  ta.edges = edges;
  ta.qs = d_qs;
  ta.qshift = qshift;
  ta.flags = spec.flags ? 1u : 0u;
  ta.key = sk;
  ta.ne = ne;
  ta.heads = TileHeads{heads, dflag + 3, (uint32_t)n_tile};
  ta.bits = bits;
  ta.bbits = bbits;
  ta.info = info;
  ta.cells = cells;
  ta.inner = inner;
  ta.flag = dflag;
  ta.front = front;
  GroupArgs ga{sk, info, level, inner, ne, qshift >= 64 ? ~0ull : ((1ull << qshift) - 1ull),
               qshift, d_qs, nullptr};
  const unsigned tile_grid =
      (unsigned)std::min<uint64_t>((n_tile + WPB - 1) / WPB, (uint64_t)num_sms() * 32);
  const unsigned crowd_grid =
      (unsigned)std::min<uint64_t>((n_tile + CROWD) / (CROWD + 1), (uint64_t)num_sms() * 4);
  if (ne) {
    element_kernel<<<grid_for(ne, 256), 256, 0, s>>>(sk, si, rval, n_rec, ne, items, pair_query,
                                                    pair_slot, d_qs, spec.B, ta.heads, info,
                                                    level, cells, rec, dflag);
    note_launch();
    if (n_tile) {
      TraceScope tr1("cover.raster", s);
      tile_raster_kernel<<<tile_grid, TPB, 0, s>>>(ta);
      note_launch();
      if (n_tile > CROWD && (Q > 1 || spec.NP > CROWD)) {
        crowd_raster_kernel<<<crowd_grid, TPB, 0, s>>>(ta);
        note_launch();
      }
    }
    group_count_kernel<<<grid_for(ne, 256), 256, 0, s>>>(ga, cnt, code, qhead, dflag, sums);
    note_launch();
    SDB_TRY_CUDA(cudaGetLastError());
    SDB_TRY(exclusive_scan<uint64_t>(cnt, off, ne, tot, s));
    SDB_TRY(exclusive_scan_u32(cells, coff, ne, tot + 1, s));
  }
  uint64_t* dqoff;
  SDB_TRY(sc.get(&dqoff, Q));
  if (ne) {
    query_offsets_kernel<<<grid_for(Q, 256), 256, 0, s>>>(qhead, Q, off, dqoff);
    note_launch();
    SDB_TRY_CUDA(cudaGetLastError());
  }
  std::vector<uint64_t> hqoff(Q, ~0ull);
  if (ne && spec.split)
    SDB_TRY_CUDA(cudaMemcpyAsync(hqoff.data(), dqoff, (size_t)Q * 8, cudaMemcpyDeviceToHost, s));
  uint64_t htot[2] = {0, 0};
  unsigned int hflag[5] = {0, 0, 0, 0, 0};
  std::vector<uint32_t> hhead(Q);
  std::vector<unsigned long long> hsums(FRONT_SPREAD + 2 * SPREAD);
  SDB_TRY_CUDA(cudaMemcpyAsync(htot, tot, 16, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaMemcpyAsync(hflag, dflag, 20, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaMemcpyAsync(hhead.data(), qhead, (size_t)Q * 4, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaMemcpyAsync(hsums.data(), front, hsums.size() * 8, cudaMemcpyDeviceToHost, s));
  SDB_TRY_CUDA(cudaStreamSynchronize(s));
  if (hflag[1] || (Q > 1 && (hflag[0] || hflag[2]))) {
    *outcome = hflag[1]   ? TileOutcome::crowded
               : hflag[2] ? TileOutcome::overlapping
                          : TileOutcome::nested;
    return SDB_OK;
  }
  unsigned long long nfront = 0;
  for (uint32_t i = 0; i < FRONT_SPREAD; ++i) nfront += hsums[i];
  GroupTotals total = group_totals(hsums.data() + FRONT_SPREAD);
  const uint64_t ncells = htot[1];
  // the limits of the refinement to the finest level
  if (4 * nfront > 0xffffffffull) {
    set_error("covering: the last level's frontier is too large (%llu cells)", nfront);
    return SDB_ENOMEM;
  }
  if (ncells >= 0xffffffffull) {
    set_error("covering: %llu cells exceed the 32-bit index range", (unsigned long long)ncells);
    return SDB_ENOMEM;
  }
  TileBase tb{};
  const bool nested = hflag[0] != 0;  // one query
  if (nested) {
    uint32_t slots = 1;
    for (uint32_t i = 0; i < spec.NP; ++i) slots = std::max(slots, spec.pair_slot[i] + 1);
    SDB_TRY_CUDA(cudaMemsetAsync(sums, 0, 2 * SPREAD * 8, s));
    SDB_TRY(nested_groups(ta, level, n_tile, spec.q[0].F, slots, sc, s, &ga, &tb));
    SDB_TRY(sc.get(&cnt, ga.ne));
    SDB_TRY(sc.get(&off, ga.ne));
    SDB_TRY(sc.get(&code, ga.ne));
    group_count_kernel<<<grid_for(ga.ne, 256), 256, 0, s>>>(ga, cnt, code, qhead, dflag, sums);
    note_launch();
    SDB_TRY_CUDA(cudaGetLastError());
    SDB_TRY(exclusive_scan<uint64_t>(cnt, off, ga.ne, tot, s));
    SDB_TRY_CUDA(cudaMemcpyAsync(htot, tot, 8, cudaMemcpyDeviceToHost, s));
    SDB_TRY_CUDA(cudaMemcpyAsync(hsums.data(), sums, 2 * SPREAD * 8, cudaMemcpyDeviceToHost, s));
    SDB_TRY_CUDA(cudaMemcpyAsync(hflag, dflag, 12, cudaMemcpyDeviceToHost, s));
    SDB_TRY_CUDA(cudaStreamSynchronize(s));
    if (hflag[1]) {
      *outcome = TileOutcome::crowded;
      return SDB_OK;
    }
    total = group_totals(hsums.data());
    hhead[0] = 0;
  }
  if (total.entries >= LIST_LIMIT) {
    set_error("covering: %llu list entries exceed the 32-bit list range",
              (unsigned long long)total.entries);
    return SDB_ENOMEM;
  }
  // entries: the groups' ranges, plus per query its sentinel, plus the empty
  // range of a query without records
  std::vector<QueryFix> hq;
  std::vector<uint64_t> hextra(Q);
  const uint64_t extra = query_fixes(hhead, ne, &hq);
  for (uint32_t q = 0; q < Q; ++q) hextra[q] = hq[q].extra;
  const uint64_t E = total.ranges + extra, nids = total.entries;
  if (E >= 0x7fffffffull) {  // entry indices travel in 31 bits of the packed payload
    set_error("covering: %llu ranges exceed the 32-bit index range", (unsigned long long)E);
    return SDB_ENOMEM;
  }
  std::vector<QueryOut> hout(Q);
  if (spec.split) {
    out->slices.assign(Q, CoverSlice{});
    uint64_t next = htot[0];
    for (uint32_t q = Q; q-- > 0;) {  // a query ends where the next one with records begins
      CoverSlice& c = out->slices[q];
      const bool any = hqoff[q] != ~0ull;
      const uint64_t at = any ? hqoff[q] : next;
      c.E = (any ? (next >> 32) - (at >> 32) : 1) + 1;
      c.nids = any ? (next & 0xffffffffull) - (at & 0xffffffffull) : 0;
      SDB_TRY(dalloc_n(&c.start, c.E, s));
      SDB_TRY(dalloc_n(&c.list_off, c.E, s));
      SDB_TRY(dalloc_n(&c.pay, c.E, s));
      SDB_TRY(dalloc_n(&c.list_ids, c.nids ? c.nids : 1, s));
      const uint64_t e0 = (at >> 32) + hextra[q];
      const uint32_t l0 = (uint32_t)at;
      hout[q] = QueryOut{c.start - e0, c.list_off - e0, c.list_ids - l0, c.pay - e0, e0, l0};
      next = at;
    }
  } else {
    SDB_TRY(dalloc_n(&out->start, E, s));
    SDB_TRY(dalloc_n(&out->list_off, E, s));
    SDB_TRY(dalloc_n(&out->pay, E, s));
    SDB_TRY(dalloc_n(&out->list_ids, nids ? nids : 1, s));
    hout.assign(Q, QueryOut{out->start, out->list_off, out->list_ids, out->pay, 0, 0});
  }
  QueryOut* dout;
  SDB_TRY(sc.get(&dout, Q));
  SDB_TRY_CUDA(cudaMemcpyAsync(dout, hout.data(), (size_t)Q * sizeof(QueryOut),
                               cudaMemcpyHostToDevice, s));
  QueryFix* dq;
  uint64_t *qopen, *dextra;
  uint32_t* qlist;
  SDB_TRY(sc.get(&dq, Q));
  SDB_TRY(sc.get(&qopen, 2 * (size_t)Q));
  SDB_TRY(sc.get(&qlist, 2 * (size_t)Q));
  SDB_TRY(sc.get(&dextra, Q));
  SDB_TRY_CUDA(cudaMemcpyAsync(dq, hq.data(), (size_t)Q * sizeof(QueryFix), cudaMemcpyHostToDevice, s));
  SDB_TRY_CUDA(cudaMemcpyAsync(dextra, hextra.data(), (size_t)Q * 8, cudaMemcpyHostToDevice, s));
  if (ne) {
    TraceScope tr1("cover.emit", s);
    const RangeOut ro{dout, qopen, qlist};
    group_emit_kernel<<<grid_for(ga.ne, 256), 256, 0, s>>>(ga, off, code, dextra, ro);
    note_launch();
    if (n_tile) {
      if (nested)
        tile_emit_kernel<true><<<tile_grid, TPB, 0, s>>>(ta, off, code, dextra, ga.lomask, tb, ro);
      else
        tile_emit_kernel<false><<<tile_grid, TPB, 0, s>>>(ta, off, code, dextra, ga.lomask, tb, ro);
      note_launch();
      if (hflag[4]) {
        if (nested)
          crowd_emit_kernel<true><<<crowd_grid, TPB, 0, s>>>(ta, off, code, dextra, ga.lomask, tb, ro);
        else
          crowd_emit_kernel<false><<<crowd_grid, TPB, 0, s>>>(ta, off, code, dextra, ga.lomask, tb, ro);
        note_launch();
      }
    }
    SDB_TRY_CUDA(cudaGetLastError());
  }
  out->E = E;
  out->nids = nids;
  out->ncells = ncells;
  return finish_queries(dq, qopen, qlist, d_qs, Q, coff, ne, ncells, dout, out, s);
}

}  // namespace sdb
