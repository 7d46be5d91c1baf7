// One warp per row, walked as an endless sequence of chunks: the cursor that produces the chunks (used by the pooling
// gather and by the GAT reduce for rows of more than a few dozen edges).
//
// A chunk is up to 32 consecutive edges of ONE row: lane i holds the source id (and weight) of edge i.  A warp asks for
// chunks two ahead of the one it reduces, so the ids of a row's first chunk, and before them the row's record, are in
// flight while the rows before it are still being reduced: the dependent trips record -> ids -> source rows, about a
// microsecond each under load, are paid once per warp instead of once per row.
//
// The list is walked from its END: the pieces of long vertices first, then whole vertices from the longest bucket down, which
// fill up the end of the launch.  Rows are handed out in claims of consecutive ones from a device counter: the p.n_pieces
// entries at the end in claims of p.piece_claim (as small as possible, so that at any time the warps work on neighbouring
// pieces), the others in claims of p.claim.  (One atomic per row would serialise on the counter: 2.9M of them cost 1.5 ms.
// Pieces dealt out in turn instead drift apart: 5 % more time on 5M vertices and 100M edges.)
//
// Included by stream.cuh (uses its StreamParams, load_meta).
#pragma once

namespace it_stream {

struct Chunk {
  int32_t idx;     // source id of edge `lane`
  float w;         // its weight (1 without weights)
  int cnt;         // edges in the chunk; 0: no chunks left
  int last;        // the row ends with this chunk
  int dest, len;   // of its row
  int owner;       // vertex the row belongs to (OWNER)
  int64_t j;       // first edge
};

template <bool WEIGHTED, bool OWNER>
struct ChunkCursor {
  const StreamParams &p;
  const int lane;
  int row, row_end;       // next row to fetch, end of the claim it lies in
  int pend;               // the claim after that one (lane 0)
  it_row_meta nm;         // the record after the current row (len 0: there is none)
  int nowner;
  int64_t j;
  int left, dest, len, owner;

  __device__ __forceinline__ ChunkCursor(const StreamParams &params, int lane_)
      : p(params), lane(lane_), nowner(0), j(0), left(0), dest(0), len(0), owner(0) {
    claim((int)blockIdx.x * (THREADS / 32) + (int)(threadIdx.x >> 5));
    fetch();
  }
  // claim number c: its rows, counted from the end of the range (fewer than 2^31 with every claim past the end)
  __device__ __forceinline__ void claim(int c) {
    const bool piece = c < p.piece_claims;
    const int end = piece ? p.n_pieces : (int)(p.row_hi - p.row_lo), size = piece ? p.piece_claim : p.claim;
    row = piece ? c * size : p.n_pieces + (c - p.piece_claims) * size;
    row_end = end - row < size ? end : row + size;
    pend = lane == 0 ? atomicAdd(p.counter, 1) : 0;
  }
  __device__ __forceinline__ void fetch() {
    if (row >= row_end) claim((int)gridDim.x * (THREADS / 32) + __shfl_sync(0xffffffffu, pend, 0));
    nm.j0 = 0; nm.len = 0; nm.dest = 0;
    if (row < row_end) {
      nm = load_meta(p.meta + (p.row_hi - 1 - row));
      if (OWNER) nowner = __ldcs(p.owner + (p.row_hi - 1 - row));
    }
    ++row;
  }
  // lane i: the edge i of the next chunk
  __device__ __forceinline__ void next(Chunk &c) {
    c.idx = 0; c.w = 1.f;
    if (left == 0) {
      if (nm.len == 0) { c.cnt = 0; return; }   // stays so: fetch() is not called again
      j = nm.j0; left = len = nm.len; dest = nm.dest; owner = nowner;
      fetch();
    }
    c.cnt = left < 32 ? left : 32;
    if (lane < c.cnt) {
      c.idx = p.indices ? __ldcs(p.indices + j + lane) : (int32_t)(j + lane);
      if (WEIGHTED) c.w = __ldcs(p.weights + j + lane);
    }
    c.j = j; c.dest = dest; c.len = len; c.owner = owner;
    j += c.cnt; left -= c.cnt;
    c.last = left == 0;
  }
};

// The walk itself.  While a stage of the current chunk is reduced the next stage is in flight: of the same chunk, or the
// first stage of the chunk after it, whichever row that belongs to.
//   next(c):              the cursor;  ahead(c): called when the chunk before c has become the current one (its ids have landed)
//   begin(c, first):      c becomes the current chunk; first: it starts a row
//   edge(k, raw):         reduce one slice of edge k of the current chunk (lanes whose slot has an edge)
//   end(c):               the current chunk ends its row
// DEEP: chunks are asked for two ahead of the current one (ahead() then finds their ids landed), else one.
template <int LPR, bool DEEP, class Warp, class Policy, class Cursor, class Ahead, class Begin, class Edge, class End>
__device__ __forceinline__ void chunk_walk(const Warp &rw, const Policy &pol, Cursor &cur, Ahead ahead, Begin begin, Edge edge, End end) {
  using G = typename Warp::G;
  constexpr int SL = G::SL, GE = G::GE, R = G::R, GB = G::GB;
  static_assert(G::S == 2, "one stage in flight, one being reduced");
  Chunk c, n, nn;
  cur.next(c);
  if (c.cnt == 0) return;   // warp-uniform
  if (DEEP) cur.next(n);
  ahead(c);
  rw.fill(pol, 0, c.idx, 0, c.cnt < GE ? c.cnt : GE);
  cp_async_commit();
  int cs = 0;
  bool first = true;
  for (;;) {
    cur.next(DEEP ? nn : n);
    begin(c, first);
    if (DEEP && n.cnt > 0) ahead(n);
    for (int k0 = 0; k0 < c.cnt; k0 += GE) {
      const int left = c.cnt - k0;
      if (left > GE) rw.fill(pol, cs ^ 1, c.idx, k0 + GE, left - GE < GE ? left - GE : GE);
      else if (n.cnt > 0) rw.fill(pol, cs ^ 1, n.idx, 0, n.cnt < GE ? n.cnt : GE);
      cp_async_commit();
      cp_async_wait<1>();
      const uint32_t sr = rw.my_ring + cs * (R * GB);
      if (left >= GE) {
#pragma unroll
        for (int u = 0; u < R; ++u) edge(k0 + u * SL + rw.slot, lds_slice<16>(sr + u * GB), true);
      } else {
        for (int u = 0; u * SL < left; ++u)   // lanes past the end read stale bytes and drop them
          edge(k0 + u * SL + rw.slot, lds_slice<16>(sr + u * GB), u * SL + rw.slot < left);
      }
      cs ^= 1;
    }
    first = c.last;
    if (c.last) end(c);
    if (n.cnt == 0) break;
    c = n;
    if (DEEP) n = nn;
  }
  cp_async_wait<0>();   // only empty groups are left
}

// The pooling gather over rows of more than a few dozen edges, one warp per row.  Bound by the source rows it keeps in
// flight; measured against walking one row at a time (record, ids and first rows fetched when the row starts):
// the same time on 128-byte rows where DRAM is the bound (5M vertices, 33..1024 edges per row: 719 against 716 us, DRAM
// at 0.73 to 0.74 of its peak), one launch for all its buckets instead of one per bucket, no spills.
#ifndef IT_CHUNK_BLOCKS
#define IT_CHUNK_BLOCKS 3       // resident CTAs per SM, and ...
#endif
#ifndef IT_CHUNK_STAGE_ROWS
#define IT_CHUNK_STAGE_ROWS 8   // ... 512-byte groups of rows per stage (four CTAs with stages of 4: GCN on 15M edges 2.76 against 2.67 ms,
#endif                          // fp32 sums on 40M 6.11 against 5.88, mean on 375M 22.4 against 22.2, 16M wide rows 3.26 against 3.20)
#ifndef IT_CHUNK_BLOCKS_PLAIN
#define IT_CHUNK_BLOCKS_PLAIN 4       // the same for 128-byte rows of graphs without pieces (launch_buckets)
#endif
#ifndef IT_CHUNK_STAGE_ROWS_PLAIN
#define IT_CHUNK_STAGE_ROWS_PLAIN 4
#endif
template <typename T, int LPR, class Policy, bool PAD, int BLOCKS, int ROWS>
__global__ void __launch_bounds__(THREADS, BLOCKS) stream_rows_chunk_kernel(StreamParams p, Policy pol) {
  extern __shared__ uint4 ring_raw[];
  const int lane = threadIdx.x & 31;
  RingWarp<T, 16, LPR, Policy, PAD, ROWS> rw;
  rw.setup((uint32_t)__cvta_generic_to_shared(ring_raw) + (uint32_t)(threadIdx.x >> 5) * (uint32_t)ring_bytes_per_warp<16, false, ROWS>(), p.src, p.src_pitch,
           p.slices, lane);
  pol.setup(lane % LPR);
  ChunkCursor<Policy::WEIGHTED, false> cur(p, lane);
  float st[Policy::NS];
  float w = 1.f;
  chunk_walk<LPR, false>(rw, pol, cur, [](Chunk &) {},
      [&](const Chunk &c, bool first) {
        w = c.w;
        if (first) {
          pol.init(st);
          if (rw.active) pol.begin_row(c.dest, 0);
        }
      },
      [&](int k, const uint4 &raw, bool valid) {
        const float we = Policy::WEIGHTED ? __shfl_sync(0xffffffffu, w, k & 31) : 1.f;
        if (valid) pol.edge(st, raw, we, 0.f);
      },
      [&](const Chunk &c) {
        rw.fold(pol, st);
        if (rw.slot == 0 && rw.active) pol.end_row(st, c.dest, 0, c.len);
      });
}

// Blocks of a launch over p.row_lo .. p.row_hi, whose last `pieces` entries are pieces of long vertices, and the rows per claim
// of the others: every block is resident from the start, a warp makes about sixteen claims, and no more than 2^18 of pieces
// altogether.
// (Row numbers fit 31 bits with every claim past the end: rows of more than 32 edges would fill the device long before.)
inline unsigned chunk_grid(StreamParams &p, int64_t pieces, int64_t max_blocks) {
  const int64_t rows = p.row_hi - p.row_lo, want = (rows + (THREADS / 32) - 1) / (THREADS / 32);
  const int64_t blocks = want < max_blocks ? want : max_blocks;
  const int64_t per = (rows - pieces) / (blocks * (THREADS / 32)) / 16;
  p.n_pieces = (int)pieces;
  p.piece_claim = (int)(1 + pieces / (1 << 18));
  p.piece_claims = (int)((pieces + p.piece_claim - 1) / p.piece_claim);
  p.claim = (int)(per < 1 ? 1 : (per > 64 ? 64 : per));
  return (unsigned)blocks;
}

}  // namespace it_stream
