// Shared by the covering builder's translation units (cover.cu, covertiles.cu).
#pragma once
#include "sdb_internal.cuh"

namespace sdb {

struct Edge {
  int32_t ax, ay, bx, by;
};

// A frontier cell of one (query, polygon) pair at level L: cell (cx, cy), its
// Hilbert id at level L and the curve's orientation (sw << 1 | cm) below it,
// so a child's id is one more digit; its edge list elist[eoff, eoff + ecnt)
// and the perturbed parity of its lower-left corner.
struct __align__(16) Item {
  uint64_t hid;
  uint32_t pair, cx, cy, eoff;
  uint32_t ecnt_par;  // edge count | parity << 31
  uint32_t orient;
};
static_assert(sizeof(Item) == 32, "two 16-byte loads per item");

// A tile is a boundary cell TILE_DEPTH levels above its query's finest level:
// 32 x 32 finest cells, a bit each in the 32 lanes of a warp.
constexpr uint32_t TILE_DEPTH = 5;
// polygons of one tile that a warp takes one after the other
constexpr uint32_t TILE_MAX_GROUP = 512;
// polygons over one another, above the tiles, that one thread sorts and compares (its
// work grows with their square; at 512 it still beats the refinement, covertiles.cu)
constexpr uint32_t MAX_OVERLAP = 512;

// per query (one thread each): its offset and record count, its sentinel
// (start 4^F), and the single empty range of a query without records
struct QueryFix {
  uint64_t extra;      // entries of earlier queries that are no ranges of groups
  uint64_t next_head;  // first record of the next query with records (or n)
  uint32_t prev;       // the last earlier query with records (or NONE)
  uint32_t head;       // the query's first record (or NONE)
};
// Where a query's ranges go: arrays indexed by the entry's number over all queries
// (a query with arrays of its own holds them moved back by e0 entries and l0 list
// entries), and what is taken off the numbers stored in them.
struct QueryOut {
  uint64_t* start;
  uint32_t* list_off;
  uint32_t* list_ids;
  uint32_t* pay;
  uint64_t e0;
  uint32_t l0;
};
// the queries' fixes from their first records (of n, 0xffffffff: none); returns
// the entries that are no ranges of groups
uint64_t query_fixes(const std::vector<uint32_t>& head, uint64_t n, std::vector<QueryFix>* out);
// sentinels, empty queries, and the slices and record counts of all queries.
// coff (nullable): records before sorted element i (n_cells in all); without it
// every element is one record.
sdb_status finish_queries(const QueryFix* dq, const uint64_t* qopen, const uint32_t* qlist,
                          const CoverQuery* d_qs, uint32_t Q, const uint64_t* coff,
                          uint64_t n_elements, uint64_t n_cells, const QueryOut* d_out,
                          CoverSet* out, cudaStream_t s);

enum class TileOutcome { made, nested, overlapping, crowded };
// The covering set from the n_rec coarse records (rkey, rval) and the n_tile
// tile items with their edge lists (covertiles.cu).  overlapping: cells of different
// polygons of one of several queries overlap at different levels inside a tile; nested:
// the same of coarser cells and whole tiles, of which a viewport may keep no cell;
// crowded: a tile meets too many polygons, or too many lie over one another; then
// nothing is made.
sdb_status cover_tiles(const uint64_t* rkey, const uint32_t* rval, uint64_t n_rec, const Item* items,
                       uint64_t n_tile, const uint32_t* elist, const Edge* edges,
                       const uint32_t* pair_query, const uint32_t* pair_slot,
                       const CoverQuery* d_qs, const CoverSpec& spec, uint32_t qshift,
                       int key_bits, cudaStream_t s, CoverSet* out, TileOutcome* outcome);

}  // namespace sdb
