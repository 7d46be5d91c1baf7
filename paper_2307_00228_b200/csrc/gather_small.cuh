// One kernel per layer for small graphs.  Some blocks walk the rows of at most 32 edges, a lane group per row, as the kernel for short
// rows does; some write the rows without edges, 32 of them per warp at a time; the others take the remaining rows, a warp per row
// (pieces of long vertices, whole vertices), source rows straight into registers, and fold the pieces of a long vertex
// in the warp that finishes the last of them.  The record of a warp's next-but-one row and the ids of its next row are in
// flight while a row is reduced.
// What bounds it: the dependent trips record -> ids -> source rows out of the L2 and the launch itself.  A layer of 10k
// vertices and 100k edges took five launches (a memset, three kernels by row length, empty rows, combine).  Measured: two fp32
// layers of that graph 150 -> 35 us; the layers of a GAT on 30k vertices and 420k edges 184 -> 63 us.
//
// Included by gather_rows.cuh and gat_rows.cuh.
#pragma once

#include "stream.cuh"

namespace it_stream {

// The pieces of long vertices in flight: the warp that finishes the last piece of a vertex folds them all.
struct PieceParams {
  const int32_t *__restrict__ piece_long;   // which long vertex a piece belongs to
  const int64_t *__restrict__ piece_ptr;
  const int32_t *__restrict__ long_owners;
  int *done;                                // pieces finished, per long vertex: zero before and after the launch
};

// All lanes of the warp have written their share of piece `slot`: true (warp-uniform) in the warp that finished the last
// piece of the vertex; the others' partial results are then visible to it (through the L2: read them with __ldcg).
__device__ __forceinline__ bool last_piece(const PieceParams &q, int slot, int lane, int &k) {
  k = __ldg(q.piece_long + slot);
  __threadfence();
  __syncwarp();
  int last = 0;
  if (lane == 0) {
    const int n = (int)(__ldg(q.piece_ptr + k + 1) - __ldg(q.piece_ptr + k));
    last = atomicAdd(q.done + k, 1) == n - 1;
    if (last) q.done[k] = 0;
  }
  last = __shfl_sync(0xffffffffu, last, 0);
  if (last) __threadfence();
  return last != 0;
}

constexpr int SMALL_BLOCKS = 3;   // resident CTAs per SM

// How a launch is shared out: the first blocks take entries [short_lo, short_hi) of the list, the next ones those before, the others
// the rest, in proportion to what they cost, since a launch is as long as its longest share.  A lane group's row costs about eight
// edges besides its own, and a warp has 32 / lpr of them at a time; a warp's row about as much as sixteen, and the more steps the more
// lanes an edge takes.  Measured against twice / half of the lane groups' share: attention, 30k vertices / 420k edges, 128-byte rows
// 63 us against 65 / 79; 30k / 400k, 512-byte rows 62 against 76 / 63; 100k / 1.8M, 256-byte rows 127 against 143 / 147; GCN, 8k / 190k,
// 128- and 64-byte rows 33 against 34 / 38.
// A row without edges costs about three (1, 2, 3, 4, 6, 9 of them: bf16 max over 768 columns, 100k vertices / 1.8M edges, power law, 2043,
// 1051, 898, 881, 880, 895 us; fp32 max over 64, 76k / 0.94M 89, 68, 71, 71, 73, 73; attention, 30k / 420k, 84, 66, 66, 66, 66, 67).  By
// lane groups or warps that take one at a time, each a trip to its record and one to its self term, the first of these took 1484 on
// blocks of their own and 1070 among the rows of all warps.
struct SmallShare {
  unsigned blocks;
  int short_blocks, empty_blocks, short_lo, short_hi, total;   // (entries [0, short_lo): rows without edges)
};
// That is the split of work that never waits for a whole row; where there are few rows for every warp, what counts is the longest warp.
// Rows that take a warp are dealt in turn, so a share of theirs that begins another round for a few rows is that much longer: then the
// lane groups get fewer blocks, or more, such that neither share is more than 12 % longer than it could be (in trips to memory: a lane
// group's row one and one per eight edges, a warp's row one and one per step).  bf16 GCN 96-64-64, 55k / 616k with hubs 66 -> 58 us (two rounds
// of pieces to one), fp32 GCN 64-128-48, 38k / 561k 94 -> 84, attention, 23k / 281k, 256-byte rows 79 -> 70, bf16 sum 128-32-64, 125k / 1.8M 146 -> 121.
// groups: lane groups take the short rows; row: what a row of theirs costs, in edges.
inline SmallShare small_share(const it_graph *g, int lpr_row, bool groups, int row) {
  SmallShare s;
  const int lpr = lpr_row < 8 ? 8 : lpr_row;
  s.total = (int)g->h_list_offsets[g->n_lists];
  s.short_lo = s.short_hi = (int)g->h_list_offsets[1];
  int64_t short_cost = 0, cost = 0;
  struct { int rows, trips; } walk[IT_MAX_BUCKETS + 1];   // lists whose rows take a warp, longest first
  int n_walk = 0;
  double short_trips = 0;   // of all lane groups
  const int step = 128 / (lpr_row < 4 ? 4 : lpr_row);   // edges in flight of a warp's row
  const int64_t empty_cost = (int64_t)s.short_lo * 3 * lpr / 16;
  for (int b = g->n_lists; b-- > 1;) {
    const int64_t rows = g->h_list_offsets[b + 1] - g->h_list_offsets[b], edges = g->h_list_edges[b];
    if (rows == 0) continue;
    if (groups && g->list_bounds[b] <= IT_SHORT_BELOW && b != g->n_lists - 1) {
      if (s.short_hi < (int)g->h_list_offsets[b + 1]) s.short_hi = (int)g->h_list_offsets[b + 1];
      short_cost += (rows * row + edges) * lpr / 16;
      // (the groups of a warp wait for the longest of their rows)
      short_trips += (double)rows * row / 8 + (g->list_bounds[b] <= IT_SHORT_EDGES ? (double)rows : (double)edges / 8 + 0.7 * (double)rows);
    } else {
      cost += rows * 16 + edges * 2 * lpr / 16;
      walk[n_walk].rows = (int)rows;
      walk[n_walk++].trips = 1 + ((int)edges / (int)rows + step - 1) / step;
    }
  }
  const int most = g->num_sms * SMALL_BLOCKS;
  const int64_t all = short_cost + cost + empty_cost;
  auto part = [&](int64_t of, int want) {   // (at least a block where there is anything to do; two are left for the others)
    int n = all > 0 ? (int)(most * of / all) : 0;
    if (n < 1 && want > 0) n = 1;
    if (n > most - 2) n = most - 2;
    return n < want ? n : want;
  };
  const int per_block = THREADS / lpr, want_short = (s.short_hi - s.short_lo + per_block - 1) / per_block;
  s.empty_blocks = part(empty_cost, (s.short_lo + THREADS / 8 - 1) / (THREADS / 8));
  s.short_blocks = part(short_cost, want_short);
  const int rest = most - s.empty_blocks;
  if (n_walk > 0 && want_short > 0) {
    const double per_group = short_trips / per_block;
    auto longest = [&](int short_blocks) {   // trips of the longest warp
      const int warps = (rest - short_blocks) * (THREADS / 32);
      int at = 0, round = 0, trips = 0;
      for (int i = 0; i < n_walk; ++i) {
        at += walk[i].rows;
        const int to = (at + warps - 1) / warps;
        trips += (to - round) * walk[i].trips;
        round = to;
      }
      return trips;
    };
    auto first = [&](auto holds) {   // the first number of short blocks in [1, rest) from which on a condition holds
      int lo = 1, hi = rest;
      while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (holds(mid)) hi = mid;
        else lo = mid + 1;
      }
      return lo;
    };
    const int cross = first([&](int x) { return per_group <= (double)x * longest(x); });   // the lane groups' is the shorter share
    double best = cross < rest ? longest(cross) : per_group / (rest - 1);
    if (cross > 1 && per_group / (cross - 1) < best) best = per_group / (cross - 1);
    best *= 1.12;
    const int most_short = first([&](int x) { return longest(x) > best; }) - 1, least_short = (int)(per_group / best) + 1;
    int n = s.short_blocks < most_short ? s.short_blocks : most_short;
    if (n < least_short) n = least_short;
    if (n > rest - 1) n = rest - 1;
    s.short_blocks = n < want_short ? n : want_short;
  }
  const int used = s.short_blocks + s.empty_blocks, left = most - used > 1 ? most - used : 1, want = (s.total - s.short_hi + THREADS / 32 - 1) / (THREADS / 32);
  s.blocks = (unsigned)(used + (want < 1 ? 1 : (want < left ? want : left)));
  return s;
}

// The rows without edges, a share of neighbours for every warp of their blocks.  rows(b, n): entries [b, b + n), n <= 32.
template <class Rows>
__device__ __forceinline__ void small_empties(const SmallShare &sh, Rows rows) {
  const int warps = sh.empty_blocks * (THREADS / 32), each = (sh.short_lo + warps - 1) / warps;
  int b = (((int)blockIdx.x - sh.short_blocks) * (THREADS / 32) + (int)(threadIdx.x >> 5)) * each;
  const int end = b + each < sh.short_lo ? b + each : sh.short_lo;
  for (; b < end; b += 32) rows(b, end - b < 32 ? end - b : 32);
}

// The rows of one warp, from the end of the list (pieces first) in turn, without the short rows.
//   row(m, idx, w): reduce one row; idx / w: ids and weights of its first 32 edges, one per lane
struct SmallRow { int j0, len, dest, owner; };   // (edges of a small graph are counted with 31 bits)
template <bool WEIGHTED, bool OWNER, class Row>
__device__ __forceinline__ void small_walk(const StreamParams &p, const SmallShare &sh, int lane, Row row) {
  const int first = sh.short_blocks + sh.empty_blocks, W = ((int)gridDim.x - first) * (THREADS / 32), n = sh.total - sh.short_hi;
  int i = ((int)blockIdx.x - first) * (THREADS / 32) + (int)(threadIdx.x >> 5);
  SmallRow m[3];
  auto fetch = [&](int at, SmallRow &x) {
    x = SmallRow{0, 0, 0, 0};
    if (at < n) {
      const int entry = sh.total - 1 - at;
      const it_row_meta r = load_meta(p.meta + entry);
      x.j0 = (int)r.j0; x.len = r.len; x.dest = r.dest;
      if (OWNER) x.owner = __ldcs(p.owner + entry);
    }
  };
  auto ids = [&](const SmallRow &x, int32_t &idx, float &w) {
    idx = 0; w = 1.f;
    if (lane < x.len) {
      idx = p.indices ? __ldg(p.indices + x.j0 + lane) : x.j0 + lane;
      if (WEIGHTED && p.weights) w = __ldg(p.weights + x.j0 + lane);
    }
  };
  int32_t idx[2];
  float w[2];
  fetch(i, m[0]);
  fetch(i + W, m[1]);
  ids(m[0], idx[0], w[0]);
  for (; i < n; i += W) {
    fetch(i + 2 * W, m[2]);
    ids(m[1], idx[1], w[1]);
    row(m[0], idx[0], w[0]);
    m[0] = m[1]; m[1] = m[2];
    idx[0] = idx[1]; w[0] = w[1];
  }
}

inline PieceParams piece_params(const it_graph *g, int *done) {
  PieceParams q;
  q.piece_long = g->piece_long; q.piece_ptr = g->piece_ptr; q.long_owners = g->long_owners; q.done = done;
  return q;
}

}  // namespace it_stream
