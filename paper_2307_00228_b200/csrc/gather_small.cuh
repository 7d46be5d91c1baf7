// One kernel per layer for small graphs.  Some blocks walk the rows of at most 32 edges and those of none, a lane group per row, as
// the kernel for short rows does; the others take the remaining rows, a warp per row (pieces of long
// vertices, whole vertices), source rows straight into registers, and fold the pieces of a long vertex
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

// How a launch is shared out: blocks [0, short_blocks) take entries [short_lo, short_hi) of the list, the others the rest, in
// proportion to what they cost, since a launch is as long as its longer share.  A lane group's row costs about eight edges besides its
// own, and a warp has 32 / lpr of them at a time; a warp's row about as much as sixteen, and the more steps the more lanes an edge
// takes.  Rows without edges, which had a warp each, cost a lane group half a row.  Measured against twice / half of the lane groups'
// share: attention, 30k vertices / 420k edges, 128-byte rows 63 us against 65 / 79; 30k / 400k, 512-byte rows 62 against 76 / 63; 100k /
// 1.8M, 256-byte rows 127 against 143 / 147; GCN, 8k / 190k, 128- and 64-byte rows 33 against 34 / 38.
struct SmallShare {
  unsigned blocks;
  int short_blocks, short_lo, short_hi, total;
};
// groups: lane groups take rows with edges too (else only those without); row: what a lane group's row costs, in edges.
inline SmallShare small_share(const it_graph *g, int lpr, bool groups, int row) {
  SmallShare s;
  s.total = (int)g->h_list_offsets[g->n_lists];
  int64_t short_cost = 0, cost = 0;
  s.short_lo = s.short_hi = 0;
  for (int b = 0; b < g->n_lists; ++b) {
    const int64_t rows = g->h_list_offsets[b + 1] - g->h_list_offsets[b], edges = g->h_list_edges[b];
    if (b == 0 || (groups && g->list_bounds[b] <= IT_SHORT_BELOW && b != g->n_lists - 1)) {
      s.short_hi = (int)g->h_list_offsets[b + 1];
      short_cost += (b == 0 ? rows * row / 2 : rows * row + edges) * lpr / 16;
    } else {
      cost += rows * 16 + edges * 2 * lpr / 16;
    }
  }
  const int rows = s.total - (s.short_hi - s.short_lo), most = g->num_sms * SMALL_BLOCKS;
  const int want_short = (int)((s.short_hi - s.short_lo + THREADS / lpr - 1) / (THREADS / lpr)), want = (rows + THREADS / 32 - 1) / (THREADS / 32);
  int share = short_cost > 0 ? (int)(most * short_cost / (short_cost + cost)) : 0;
  if (share < 1 && want_short > 0) share = 1;
  if (share > most - 1) share = most - 1;
  s.short_blocks = share < want_short ? share : want_short;
  const int left = most - s.short_blocks;
  s.blocks = (unsigned)(s.short_blocks + (want < 1 ? 1 : (want < left ? want : left)));
  return s;
}

// The rows of one warp, from the end of the list (pieces first) in turn, without the short rows.
//   row(m, idx, w): reduce one row; idx / w: ids and weights of its first 32 edges, one per lane
struct SmallRow { int j0, len, dest, owner; };   // (edges of a small graph are counted with 31 bits)
template <bool WEIGHTED, bool OWNER, class Row>
__device__ __forceinline__ void small_walk(const StreamParams &p, const SmallShare &sh, int lane, Row row) {
  const int W = ((int)gridDim.x - sh.short_blocks) * (THREADS / 32), above = sh.total - sh.short_hi, n = above + sh.short_lo;
  int i = ((int)blockIdx.x - sh.short_blocks) * (THREADS / 32) + (int)(threadIdx.x >> 5);
  SmallRow m[3];
  auto fetch = [&](int at, SmallRow &x) {
    x = SmallRow{0, 0, 0, 0};
    if (at < n) {
      const int entry = at < above ? sh.total - 1 - at : n - 1 - at;
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
