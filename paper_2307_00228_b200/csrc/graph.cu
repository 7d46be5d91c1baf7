// Graph ingest, validation, hub split into shadow rows, degree buckets.
// Integer-only work.  The arrays that the interface reports are a pure function of (indptr, threshold) and reproducible bit for
// bit; in the lists that the gather walks the order of the pieces inside a bin is that of atomics, which no result depends on.
#include <mutex>
#include <new>
#include <type_traits>
#include <stdarg.h>
#include <string.h>

#include "common.cuh"

// ----------------------------------------------------------------------------- error text
static thread_local char g_err[512] = "";
void it_set_error(const char *fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
}
extern "C" const char *it_last_error_message(void) { return g_err; }
extern "C" const char *it_status_string(it_status s) {
  switch (s) {
    case IT_OK: return "IT_OK";
    case IT_ERR_INVALID_ARG: return "IT_ERR_INVALID_ARG";
    case IT_ERR_BAD_GRAPH: return "IT_ERR_BAD_GRAPH";
    case IT_ERR_UNSUPPORTED: return "IT_ERR_UNSUPPORTED";
    case IT_ERR_WORKSPACE: return "IT_ERR_WORKSPACE";
    case IT_ERR_OOM: return "IT_ERR_OOM";
    case IT_ERR_CUDA: return "IT_ERR_CUDA";
    case IT_ERR_TIMEOUT: return "IT_ERR_TIMEOUT";
  }
  return "IT_ERR_?";
}

// ----------------------------------------------------------------------------- indptr access
struct IndptrView {
  const void *p;
  int is64;
  __device__ __forceinline__ int64_t operator[](int64_t i) const {
    return is64 ? reinterpret_cast<const int64_t *>(p)[i]
                : (int64_t) reinterpret_cast<const int32_t *>(p)[i];
  }
};

__device__ __forceinline__ int64_t groups_of(int64_t d, int64_t T) {
  return (T <= 0 || d <= T) ? 1 : (d + T - 1) / T;
}

// ----------------------------------------------------------------------------- validation
// bit 0: indptr[0] != 0, bit 1: indptr decreasing, bit 2: indptr[n] != e, bit 3: source out of range
__global__ void validate_indptr_kernel(IndptrView ip, int64_t n, int64_t e, int *flags) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  int bad = 0;
  if (i == 0) {
    if (ip[0] != 0) bad |= 1;
    if (ip[n] != e) bad |= 4;
  }
  if (i < n && ip[i + 1] < ip[i]) bad |= 2;
  if (bad) atomicOr(flags, bad);
}

// Four ids per load (`head` ids up to the first 16-byte boundary and the last few on their own): bound by reading them.
// Runs after validate_indptr_kernel and reads no id of an indptr that failed: `e` is then no count of ids that the caller holds.
__global__ void __launch_bounds__(256) validate_indices_kernel(const int32_t *__restrict__ idx, int64_t e, int64_t n, int head, int *flags) {
  if (*reinterpret_cast<volatile int *>(flags) != 0) return;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const uint32_t top = (uint32_t)n;   // n < 2^31: a negative id is a large unsigned one
  bool bad = false;
  const int4 *v = reinterpret_cast<const int4 *>(idx + head);
  const int64_t quads = (e - head) / 4;
  for (int64_t i = first; i < quads; i += 4 * stride) {
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u * stride < quads) {
        const int4 x = __ldcs(v + i + u * stride);
        bad |= (uint32_t)x.x >= top || (uint32_t)x.y >= top || (uint32_t)x.z >= top || (uint32_t)x.w >= top;
      }
  }
  for (int64_t i = first; i < head; i += stride) bad |= (uint32_t)idx[i] >= top;
  for (int64_t i = head + quads * 4 + first; i < e; i += stride) bad |= (uint32_t)idx[i] >= top;
  if (bad) atomicOr(flags, 8);
}

// ----------------------------------------------------------------------------- split
// The shadow rows and the degree buckets in one pass over the vertices: count per tile, scan the tile counts, emit.
// Every vertex adds rows to at most two buckets (all groups of a split vertex hold d / ng or d / ng + 1 edges), so the row
// numbers, the list of long vertices and the positions inside every bucket are prefix sums of the same pass: columns
// 0 .. nb - 1 the buckets, nb the rows, nb + 1 the split vertices, nb + 2 the long vertices, nb + 3 their pieces, and from
// nb + 4 on the lists that the gather walks.
//
// The gather does not walk the shadow rows of a hub but finer pieces of its segment, and pieces of every vertex of more than
// long_above edges (1024 to 4096, whatever T is): those of all such vertices are ordered by where in its vertex's segment a piece lies.  Where source ids ascend
// inside a segment, as a sorted edge list has them, pieces at the same relative position read the same part of the source table, and
// those that are in flight together share it through the L2 cache.  (Without that order they cost nothing either: 2M vertices, 40M
// edges in random order, bf16 mean 920 -> 926 us, GAT 2511 -> 2393, fp32 sums 2333 -> 2215.)  Whole passes, against
// one block per row of up to T edges in vertex order: 5M vertices / 100M edges, GAT, 13.1 -> 11.7 ms; 20M / 200M with 100 hubs
// of 1M edges, max pooling, 20.0 -> 17.4; 2M / 40M, fp32 sums, 6.6 -> 5.95; 25M / 375M, mean, 23.3 -> 22.6.
// A piece is a 64th of its vertex (it then spans a 64th of the table), at least 128 edges (its fp32 partial result costs a row
// written and a row read: 3 % of 128 rows; 64 and 32 edges cost 1 to 2 % more on GAT) and at most 512 (one warp walks it), more only
// where a vertex would have more than PIECES_MOST of them (one block folds them: a single vertex of 20M edges 556 -> 325 us).
// Source tables of fewer than 2^17 rows fit the cache whatever the order: pieces of at least 256 edges.
// Bound by reading indptr twice and writing 36 bytes per row; a scan per bucket (each over every row, three launches with a
// read of two 8-byte bounds per row) took 3.2 ms of device time for 5M vertices and six buckets, this one 3.0 with
// everything around it (create + split: 14.3 -> 2.4 ms on a quiet machine, 0.5 of it kernels; the derived arrays are one allocation
// instead of nine, which the split after the create reuses.  cudaMalloc and cudaFree take 0.4 ms each there and several on a busy one.)
constexpr int SPLIT_THREADS = 256;
constexpr int SPLIT_ITEMS = 8;                                    // vertices per lane
constexpr int SPLIT_TILE = 32 * SPLIT_ITEMS;                      // a tile is one warp's 256 consecutive vertices
constexpr int SPLIT_COLS = 2 * IT_MAX_BUCKETS + 4;
constexpr int N_FIXED = 5;                                        // bounds of the buckets below T, of the lists below long_above
constexpr int N_LISTS = N_FIXED + 1;                              // lists of whole vertices
constexpr int64_t PIECES_MOST = 8192;                             // of one vertex (or one more): one block or warp folds them
constexpr int PIECE_BINS = 256;                                   // steps of the order in which pieces are walked

struct Bounds { int64_t b[IT_MAX_BUCKETS]; int nb; };
__device__ __forceinline__ int bucket_of(int64_t len, const Bounds &B) {
  int k = 0;
  while (k < B.nb - 1 && len > B.b[k]) ++k;
  return k;
}

// The list of a vertex that is gathered whole: bounds 0, 8, 32, 256, 1024, long_above.  For a vertex of at most T edges it has the
// number of its bucket (whose bounds are those of these below T, then T).
__device__ __forceinline__ int list_of(int64_t len) { return (len > 0) + (len > 8) + (len > 32) + (len > 256) + (len > 1024); }

struct LongInfo { int64_t r0, pos_a, pos_b; };   // a long vertex: its first row; bucket positions of its longer / shorter groups

struct SplitParams {
  IndptrView ip;
  int64_t n, e, T;
  Bounds B;
  int64_t n_tiles;
  int64_t *tiles;          // [SPLIT_COLS][n_tiles]
  int64_t *totals;         // [SPLIT_COLS] column sums, then [IT_MAX_BUCKETS] edges per list (the last one: of the pieces)
  int64_t long_above;      // vertices of more edges are gathered in pieces
  int piece_min, piece_max;
  int64_t *shadow_indptr; int32_t *shadow_owner; int64_t *owner_indptr;
  int64_t *bucket_offsets; int32_t *bucket_rows;
  it_row_meta *list_meta; int32_t *list_owner;
  int32_t *long_owners; int64_t *piece_ptr; int32_t *piece_long; LongInfo *info;   // [long vertices]
  int *bins;               // [2][PIECE_BINS]: pieces per bin, then the next free place
};

__device__ __forceinline__ int64_t pieces_of(int64_t d, const SplitParams &p) {
  const int64_t by_share = d / 64, least = by_share < p.piece_min ? p.piece_min : by_share, most = least > p.piece_max ? p.piece_max : least;
  const int64_t len = d / PIECES_MOST > most ? d / PIECES_MOST : most;
  return (d + len - 1) / len;
}

// What a vertex adds: ng rows; `rem` of them in bucket ka (one edge longer), the others in bucket kb.
struct VertexRows { int64_t ng, rem; int ka, kb; };
__device__ __forceinline__ VertexRows rows_of(int64_t d, const SplitParams &p) {
  VertexRows r;
  r.ng = groups_of(d, p.T);
  if (r.ng == 1) {
    r.rem = 0;
    r.ka = r.kb = bucket_of(d, p.B);
  } else {
    const int64_t base = d / r.ng;
    r.rem = d % r.ng;
    r.ka = bucket_of(base + 1, p.B);
    r.kb = bucket_of(base, p.B);
  }
  return r;
}

// Lane c of a warp keeps column c.  One step over 32 vertices; `mine`: lane of bucket or list k: the vertices in bucket k.
__device__ __forceinline__ unsigned bucket_mask(int kb, int nb, int lane) {
  unsigned mine = 0;
  for (int k = 0; k < nb; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, kb == k);
    if (lane == k || lane == nb + 4 + k) mine = m;
  }
  return mine;
}
// vertices `plain`, gathered whole
__device__ __forceinline__ void add_plain(int64_t &col, unsigned mine, unsigned plain, int nb, int lane) {
  if (lane == nb) col += __popc(plain);
  else col += __popc(mine & plain);   // (0 for the columns of long vertices)
}
// vertex l, of several groups or gathered in pieces (np > 0; else whole, from list kl)
struct LongCols { int64_t ng, rem, np; int ka, kb, kl; };
__device__ __forceinline__ LongCols long_cols(int64_t d, const VertexRows &r, int l, const SplitParams &p) {
  LongCols c;
  c.ng = __shfl_sync(0xffffffffu, r.ng, l); c.rem = __shfl_sync(0xffffffffu, r.rem, l);
  c.ka = __shfl_sync(0xffffffffu, r.ka, l); c.kb = __shfl_sync(0xffffffffu, r.kb, l);
  const int64_t dl = __shfl_sync(0xffffffffu, d, l);
  c.np = dl > p.long_above ? pieces_of(dl, p) : 0;
  c.kl = list_of(dl);
  return c;
}
__device__ __forceinline__ void add_long(int64_t &col, const LongCols &c, int nb, int lane) {
  if (lane == c.ka) col += c.rem;
  if (lane == c.kb) col += c.ng - c.rem;
  if (lane == nb) col += c.ng;
  if (lane == nb + 1 && c.ng > 1) col += 1;
  if (lane == nb + 2 && c.np > 0) col += 1;
  if (lane == nb + 3) col += c.np;
  if (lane == nb + 4 + c.kl && c.np == 0) col += 1;
}
// vertices that take their turn one by one: of several groups, or gathered in pieces
__device__ __forceinline__ bool one_by_one(int64_t d, const VertexRows &r, const SplitParams &p) { return r.ng > 1 || d > p.long_above; }

__global__ void __launch_bounds__(SPLIT_THREADS) split_count_kernel(SplitParams p) {
  __shared__ unsigned long long edges[IT_MAX_BUCKETS];
  const int lane = threadIdx.x & 31, nb = p.B.nb;
  if (threadIdx.x < IT_MAX_BUCKETS) edges[threadIdx.x] = 0;
  __syncthreads();
  const int64_t tile = (int64_t)blockIdx.x * (SPLIT_THREADS / 32) + (threadIdx.x >> 5);
  const int64_t v0 = tile * SPLIT_TILE + lane;
  int64_t col = 0, my_edges = 0;
  int64_t d[SPLIT_ITEMS];
#pragma unroll
  for (int i = 0; i < SPLIT_ITEMS; ++i) {
    const int64_t v = v0 + i * 32;
    d[i] = v < p.n ? p.ip[v + 1] - p.ip[v] : 0;
  }
#pragma unroll
  for (int i = 0; i < SPLIT_ITEMS; ++i) {
    const VertexRows r = rows_of(d[i], p);
    const unsigned valid = __ballot_sync(0xffffffffu, v0 + i * 32 < p.n), mine = bucket_mask(r.kb, nb, lane);
    unsigned lng = __ballot_sync(0xffffffffu, one_by_one(d[i], r, p));
    add_plain(col, mine, valid & ~lng, nb, lane);
    while (lng) {   // rare
      const int l = __ffs(lng) - 1;
      lng &= lng - 1;
      add_long(col, long_cols(d[i], r, l, p), nb, lane);
    }
    const int kl = list_of(d[i]);
#pragma unroll
    for (int k = 1; k < N_LISTS; ++k) {   // whole vertices have at most 4096 edges: 32-bit sums
      const unsigned sum = __reduce_add_sync(0xffffffffu, kl == k && d[i] <= p.long_above ? (unsigned)d[i] : 0u);
      if (lane == k) my_edges += sum;
    }
    if (d[i] > p.long_above) atomicAdd(&edges[IT_MAX_BUCKETS - 1], (unsigned long long)d[i]);
  }
  if (lane < nb + 4 + N_LISTS && tile < p.n_tiles) p.tiles[lane * p.n_tiles + tile] = col;
  if (lane < N_LISTS && my_edges) atomicAdd(&edges[lane], (unsigned long long)my_edges);
  __syncthreads();
  if (threadIdx.x < IT_MAX_BUCKETS && edges[threadIdx.x])
    atomicAdd(reinterpret_cast<unsigned long long *>(p.totals + SPLIT_COLS + threadIdx.x), edges[threadIdx.x]);
}

__device__ __forceinline__ int64_t block_exclusive_scan(int64_t x, int64_t *total, int64_t *smem /*[33]*/) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  int64_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  __syncthreads();  // smem may still be read from a previous call
  if (lane == 31) smem[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int64_t w = lane < nwarps ? smem[lane] : 0;
    int64_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += y;
    }
    if (lane < nwarps) smem[lane] = wi - w;  // exclusive warp offsets
    if (lane == 31) smem[32] = wi;           // block total
  }
  __syncthreads();
  *total = smem[32];
  return smem[warp] + incl - x;
}

// One block per column: exclusive scan of its tile counts in place, four tiles per thread and step; the sum to totals.
__global__ void __launch_bounds__(1024) split_scan_kernel(SplitParams p) {
  __shared__ int64_t smem[33];
  int64_t *t = p.tiles + blockIdx.x * p.n_tiles;
  int64_t carry = 0;
  for (int64_t base = 0; base < p.n_tiles; base += 4096) {
    const int64_t i = base + 4 * (int64_t)threadIdx.x;
    int64_t x[4], sum = 0, total;
#pragma unroll
    for (int u = 0; u < 4; ++u) { x[u] = i + u < p.n_tiles ? t[i + u] : 0; sum += x[u]; }
    int64_t ex = carry + block_exclusive_scan(sum, &total, smem);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (i + u < p.n_tiles) t[i + u] = ex;
      ex += x[u];
    }
    carry += total;
  }
  if (threadIdx.x == 0) p.totals[blockIdx.x] = carry;
}

__global__ void __launch_bounds__(SPLIT_THREADS) split_emit_kernel(SplitParams p) {
  const int lane = threadIdx.x & 31, nb = p.B.nb;
  const unsigned below = (1u << lane) - 1u;
  const int64_t tile = (int64_t)blockIdx.x * (SPLIT_THREADS / 32) + (threadIdx.x >> 5);
  if (tile >= p.n_tiles) return;   // whole warps
  const int64_t v0 = tile * SPLIT_TILE + lane;
  int64_t j0[SPLIT_ITEMS];
  int64_t d[SPLIT_ITEMS];
#pragma unroll
  for (int i = 0; i < SPLIT_ITEMS; ++i) {
    const int64_t v = v0 + i * 32;
    j0[i] = v < p.n ? p.ip[v] : 0;
    d[i] = v < p.n ? p.ip[v + 1] - j0[i] : 0;
  }
  // lane c: the running value of column c; for a bucket or list counted from the start of all of them
  int64_t run = 0;
  if (lane < nb + 4 + N_LISTS) {
    run = p.tiles[lane * p.n_tiles + tile];
    const int first = lane < nb ? 0 : (lane >= nb + 4 ? nb + 4 : lane);
    for (int k = first; k < lane; ++k) run += p.totals[k];
  }
  if (tile == 0) {
    if (lane <= nb) {
      int64_t off = 0;
      for (int k = 0; k < lane; ++k) off += p.totals[k];
      p.bucket_offsets[lane] = off;
    }
    if (lane == 0) {
      p.shadow_indptr[p.totals[nb]] = p.e;
      p.owner_indptr[p.n] = p.totals[nb];
      p.piece_ptr[p.totals[nb + 2]] = p.totals[nb + 3];
    }
  }
#pragma unroll
  for (int i = 0; i < SPLIT_ITEMS; ++i) {
    const int64_t v = v0 + i * 32;
    const VertexRows r = rows_of(d[i], p);
    const bool is_long = d[i] > p.long_above;
    const unsigned lng = __ballot_sync(0xffffffffu, one_by_one(d[i], r, p)), mine = bucket_mask(r.kb, nb, lane);
    const unsigned same = __match_any_sync(0xffffffffu, r.kb);
    unsigned todo = __ballot_sync(0xffffffffu, v < p.n);
    int64_t row = 0, pos = 0, at = 0;   // first row; position in the buckets / in the lists
    for (;;) {   // the whole vertices up to the next long one, then that one
      const unsigned longs = lng & todo;
      const int l = longs ? __ffs(longs) - 1 : 32;
      const unsigned plain = l == 32 ? todo : todo & ((1u << l) - 1u);
      const int64_t at_row = __shfl_sync(0xffffffffu, run, nb), at_bucket = __shfl_sync(0xffffffffu, run, r.kb);
      const int64_t at_list = __shfl_sync(0xffffffffu, run, nb + 4 + r.kb);
      if ((plain >> lane) & 1u) {
        row = at_row + __popc(plain & below);
        pos = at_bucket + __popc(plain & same & below);
        at = at_list + __popc(plain & same & below);
      }
      add_plain(run, mine, plain, nb, lane);
      if (l == 32) break;
      const LongCols c = long_cols(d[i], r, l, p);
      const int64_t l_row = __shfl_sync(0xffffffffu, run, nb), l_k = __shfl_sync(0xffffffffu, run, nb + 2);
      const int64_t l_piece = __shfl_sync(0xffffffffu, run, nb + 3), l_a = __shfl_sync(0xffffffffu, run, c.ka);
      const int64_t l_b = __shfl_sync(0xffffffffu, run, c.kb) + (c.ka == c.kb ? c.rem : 0);
      const int64_t l_at = __shfl_sync(0xffffffffu, run, nb + 4 + c.kl);
      if (lane == l) {
        row = l_row; pos = l_b; at = l_at;
        if (is_long) {
          p.long_owners[l_k] = (int32_t)v;
          p.piece_ptr[l_k] = l_piece;
          p.info[l_k] = LongInfo{l_row, l_a, l_b};
        }
      }
      if (c.np == 0) {   // its groups (those of long vertices: long_rows_kernel)
        const int64_t s0 = __shfl_sync(0xffffffffu, j0[i], l), base = __shfl_sync(0xffffffffu, d[i], l) / c.ng;
        const int32_t owner = (int32_t)(v - lane + l);
        for (int64_t g = lane; g < c.ng; g += 32) {
          p.shadow_indptr[l_row + g] = s0 + g * base + (g < c.rem ? g : c.rem);
          p.shadow_owner[l_row + g] = owner;
          p.bucket_rows[g < c.rem ? l_a + g : l_b + (g - c.rem)] = (int32_t)(l_row + g);
        }
      }
      add_long(run, c, nb, lane);
      todo &= ~((2u << l) - 1u);   // (l = 31: 2u << 31 = 0, nothing left)
    }
    if (v < p.n) {
      p.owner_indptr[v] = row;
      if (r.ng == 1) {
        p.shadow_indptr[row] = j0[i];
        p.shadow_owner[row] = (int32_t)v;
        p.bucket_rows[pos] = (int32_t)row;
      }
      if (!is_long) {
        it_row_meta m;
        m.j0 = j0[i]; m.len = (int32_t)d[i]; m.dest = (int32_t)v;
        p.list_meta[at] = m;
        p.list_owner[at] = (int32_t)v;
      }
    }
  }
}

// pieces [first, last) of a vertex with np of them lie in bin b of the order
__device__ __forceinline__ int64_t bin_first(int64_t b, int64_t np) { return (b * np + PIECE_BINS - 1) / PIECE_BINS; }

// Long vertices, one block each (grid-stride).  Shadow rows by closed form
//   start(g) = indptr[v] + g * base + min(g, rem),  base = d / ng, rem = d % ng;
// and how many of its pieces lie in every bin.
__global__ void __launch_bounds__(PIECE_BINS) long_rows_kernel(SplitParams p) {
  const int64_t n_long = p.totals[p.B.nb + 2];
  int in_bin = 0;   // thread = bin
  for (int64_t k = blockIdx.x; k < n_long; k += gridDim.x) {
    const int64_t v = p.long_owners[k], s = p.ip[v], d = p.ip[v + 1] - s;
    const LongInfo f = p.info[k];
    const int64_t ng = groups_of(d, p.T), base = d / ng, rem = d % ng;
    if (ng > 1)
      for (int64_t g = threadIdx.x; g < ng; g += blockDim.x) {
        const int64_t row = f.r0 + g;
        p.shadow_indptr[row] = s + g * base + (g < rem ? g : rem);
        p.shadow_owner[row] = (int32_t)v;
        p.bucket_rows[g < rem ? f.pos_a + g : f.pos_b + (g - rem)] = (int32_t)row;
      }
    const int64_t np = p.piece_ptr[k + 1] - p.piece_ptr[k];
    in_bin += (int)(bin_first(threadIdx.x + 1, np) - bin_first(threadIdx.x, np));
  }
  if (in_bin > 0) atomicAdd(p.bins + threadIdx.x, in_bin);
}

// The pieces, bin after bin behind the lists of whole vertices.  (Inside a bin the order of the blocks is that of
// their atomics: it decides when a piece is walked, not what it holds or where its result goes.)
__global__ void __launch_bounds__(PIECE_BINS) long_pieces_kernel(SplitParams p) {
  __shared__ int64_t smem[33];
  const int64_t n_long = p.totals[p.B.nb + 2], first_piece = p.n - n_long;
  int64_t total;
  int64_t pos = first_piece + block_exclusive_scan(p.bins[threadIdx.x], &total, smem);
  int in_bin = 0;
  for (int64_t k = blockIdx.x; k < n_long; k += gridDim.x) {
    const int64_t np = p.piece_ptr[k + 1] - p.piece_ptr[k];
    in_bin += (int)(bin_first(threadIdx.x + 1, np) - bin_first(threadIdx.x, np));
  }
  if (in_bin > 0) pos += atomicAdd(p.bins + PIECE_BINS + threadIdx.x, in_bin);   // this block's share of the bin
  for (int64_t k = blockIdx.x; k < n_long; k += gridDim.x) {
    const int64_t v = p.long_owners[k], s = p.ip[v], d = p.ip[v + 1] - s;
    const int64_t p0 = p.piece_ptr[k], np = p.piece_ptr[k + 1] - p0, base = d / np, rem = d % np;
    const int64_t g0 = bin_first(threadIdx.x, np), g1 = bin_first(threadIdx.x + 1, np);
    for (int64_t g = g0; g < g1; ++g, ++pos) {
      it_row_meta m;
      m.j0 = s + g * base + (g < rem ? g : rem);
      m.len = (int32_t)(base + (g < rem ? 1 : 0));
      m.dest = (int32_t)~(p0 + g);
      p.list_meta[pos] = m;
      p.list_owner[pos] = (int32_t)v;
      p.piece_long[p0 + g] = (int32_t)k;
    }
  }
}

// ----------------------------------------------------------------------------- host side
// Status words of graphs: the validation's flags, later set by a kernel that gives up a wait.  They come from a fixed array, since an
// allocation of four bytes costs as much as any (0.33 ms, and 0.26 to give it back: a quarter of the set-up of 5M vertices / 100M edges); beyond
// that many graphs on a device at a time, and on devices beyond the first 64, a word is allocated.  A word is given back when nothing on the
// device uses it any more: after the graph's arrays, whose release waits for the device, or after a wait for the stream; where there was
// neither (`quiet` false) it stays taken, since what is still queued may write it.
constexpr int STATUS_WORDS = 1024;
static __device__ int g_status_words[STATUS_WORDS];
namespace {
constexpr int kMaxDevices = 64;
std::mutex g_status_mu;
int *g_status_base[kMaxDevices] = {nullptr};
uint64_t g_status_taken[kMaxDevices][STATUS_WORDS / 64] = {};
}  // namespace

static it_status status_take(int device, int **out) {
  if (device >= 0 && device < kMaxDevices) {
    std::lock_guard<std::mutex> lk(g_status_mu);
    if (!g_status_base[device]) {
      void *p = nullptr;
      IT_CUDA_TRY(cudaGetSymbolAddress(&p, g_status_words));
      g_status_base[device] = static_cast<int *>(p);
    }
    for (int i = 0; i < STATUS_WORDS / 64; ++i) {
      uint64_t &taken = g_status_taken[device][i];
      if (taken == ~(uint64_t)0) continue;
      const int bit = __builtin_ctzll(~taken);
      taken |= (uint64_t)1 << bit;
      *out = g_status_base[device] + i * 64 + bit;
      return IT_OK;
    }
  }
  IT_CUDA_TRY(cudaMalloc(out, sizeof(int)));
  return IT_OK;
}
static void status_give_back(int device, int *word, bool quiet) {
  if (device >= 0 && device < kMaxDevices) {
    std::lock_guard<std::mutex> lk(g_status_mu);
    const int64_t at = g_status_base[device] ? word - g_status_base[device] : -1;
    if (at >= 0 && at < STATUS_WORDS) {
      if (quiet) g_status_taken[device][at / 64] &= ~((uint64_t)1 << (at % 64));
      return;
    }
  }
  cudaFree(word);
}

// Nothing on the device may still use the graph's arrays: cudaFree waits for it.  (It may also be called while another thread
// captures a stream, which a synchronisation of the device may not.)
static void slab_free(it_graph *g) {
  cudaFree(g->slab);
  g->slab = nullptr;
  g->slab_bytes = 0;
}

static void forget_split(it_graph *g) {
  g->shadow_indptr = nullptr; g->shadow_owner = nullptr; g->owner_indptr = nullptr;
  g->long_owners = nullptr; g->piece_ptr = nullptr; g->piece_long = nullptr; g->bucket_offsets = nullptr; g->bucket_rows = nullptr;
  g->list_meta = nullptr; g->list_owner = nullptr;
  g->n_rows = g->n_split_owners = g->n_partial_rows = g->n_long = 0;
  g->n_buckets = g->n_lists = 0;
}

// The derived arrays and the scratch of a split with at most R rows, L long vertices and P pieces, carved out of one
// allocation that the graph keeps for its next split (NULL slab: only the size).
static size_t carve_split(SplitParams &p, char *slab, int64_t R, int64_t L, int64_t P) {
  size_t off = 0;
  auto take = [&](auto *&ptr, int64_t count) {
    ptr = reinterpret_cast<std::remove_reference_t<decltype(ptr)>>(slab + off);
    off += it_align_up((size_t)(count > 0 ? count : 1) * sizeof(*ptr));
  };
  take(p.totals, SPLIT_COLS + IT_MAX_BUCKETS);
  take(p.bins, 2 * PIECE_BINS);   // next to the totals: cleared with them
  take(p.tiles, SPLIT_COLS * p.n_tiles);
  take(p.bucket_offsets, IT_MAX_BUCKETS + 1);
  take(p.owner_indptr, p.n + 1);
  take(p.shadow_indptr, R + 1);
  take(p.shadow_owner, R);
  take(p.bucket_rows, R);
  take(p.list_meta, p.n + P);
  take(p.list_owner, p.n + P);
  take(p.long_owners, L);
  take(p.piece_ptr, L + 1);
  take(p.piece_long, P);
  take(p.info, L);
  return off;
}

// What a split of the graph at threshold T looks like: its parameters and how much room its arrays need at most.
struct SplitPlan {
  SplitParams p{};
  unsigned blocks;
  int64_t R, L, P;      // shadow rows, long vertices, pieces
  bool count_first;     // counted before the arrays are laid out
};
constexpr int64_t kFixedBounds[N_FIXED] = {0, 8, 32, 256, 1024};   // (list_of)

static void plan_split(const it_graph *g, int64_t T, SplitPlan &s) {
  SplitParams &p = s.p;
  const int64_t n = g->n;
  p.ip = IndptrView{g->indptr, g->indptr_type == IT_I64};
  p.n = n; p.e = g->e; p.T = T;
  p.n_tiles = (n + SPLIT_TILE - 1) / SPLIT_TILE;
  s.blocks = (unsigned)((p.n_tiles + SPLIT_THREADS / 32 - 1) / (SPLIT_THREADS / 32));
  // degree buckets: {0, 8, 32, 256, 1024, everything longer}
  p.B.nb = 0;
  for (int i = 0; i < N_FIXED; ++i)
    if (T <= 0 || kFixedBounds[i] < T) p.B.b[p.B.nb++] = kFixedBounds[i];
  p.B.b[p.B.nb++] = T > 0 ? T : INT64_MAX;

  // A piece spans 128 / d of the source table, which has to stay small against the cache: the larger the table, the longer
  // the vertices that are worth it (25M sources: pieces above 1024 edges 26.3 ms, above 4096 22.9, above 2048 22.6; 5M: above 1024
  // 11.7, above 2441 12.1).
  p.long_above = g->n_src / 12288 < 1024 ? 1024 : (g->n_src / 12288 > 4096 ? 4096 : g->n_src / 12288);
  p.piece_min = g->n_src < ((int64_t)1 << 17) ? 256 : 128;
  p.piece_max = 512;
  // Small graphs: a warp's longest row is the time of the launch, so pieces are shorter where 24 warps per SM have at most 64 edges each
  // (64 against 128 edges: 10k vertices / 100k edges 35.1 against 39.4 us, GAT 10k / 150k 24.7 / 26.8, 1000 / 150k of 2 KB rows 197 / 215;
  // beyond, 10k / 300k 47.5 / 44.4, GAT 30k / 420k 82.5 / 78.7).
  if (it_small_graph(g)) p.long_above = p.piece_min = p.piece_max = g->e <= 64 * 24 * (int64_t)g->num_sms ? 64 : 128;

  // at most one row per vertex and one more per T edges, a long vertex per long_above edges, a piece per piece_min of them
  // and one more each; only where that is far above the number of vertices are they counted before the arrays are laid out
  const int64_t e = g->e;
  s.R = n + (T > 0 ? e / T : 0); s.L = n < e / p.long_above ? n : e / p.long_above; s.P = e / p.piece_min + s.L;
  s.count_first = s.R + s.P > n + n / 2 + (1 << 22) || s.R > (int64_t)INT32_MAX - 1;
}

// Grow the graph's allocation; what it holds is not kept.
static it_status reserve(it_graph *g, size_t bytes) {
  if (bytes <= g->slab_bytes) return IT_OK;
  slab_free(g);
  size_t room = bytes + bytes / 8;   // for the few more rows of another threshold, where the device has it
  if (cudaMalloc(&g->slab, room) != cudaSuccess) {
    cudaGetLastError();
    g->slab = nullptr;
    room = bytes;
    IT_CUDA_TRY(cudaMalloc(&g->slab, room));
  }
  g->slab_bytes = room;
  return IT_OK;
}

static it_status split_impl(it_graph *g, int64_t T, cudaStream_t st) {
  // The arrays of the previous split are written over.  Where nothing but that split itself, which waited for its stream, has
  // used them this needs no wait; else what still reads them, on any stream, comes first.
  if (g->used.exchange(false)) slab_free(g);
  forget_split(g);
  g->threshold = T > 0 ? T : 0;
  const int64_t n = g->n;
  SplitPlan plan;
  plan_split(g, T, plan);
  SplitParams &p = plan.p;
  const unsigned split_blocks = plan.blocks;
  int64_t R = plan.R, L = plan.L, P = plan.P;
  const bool count_first = plan.count_first;
  int64_t h[SPLIT_COLS + IT_MAX_BUCKETS] = {0};
  auto count = [&]() -> it_status {
    IT_CUDA_TRY(cudaMemsetAsync(p.totals, 0, (size_t)((char *)p.tiles - (char *)p.totals), st));
    if (n > 0) {
      IT_LAUNCH(IT_K_SPLIT_SCAN, 0, 0, st, split_count_kernel<<<split_blocks, SPLIT_THREADS, 0, st>>>(p));
      IT_LAUNCH(IT_K_SPLIT_SCAN, 0, 0, st, split_scan_kernel<<<(unsigned)(p.B.nb + 4 + N_LISTS), 1024, 0, st>>>(p));
    }
    IT_CUDA_TRY(cudaGetLastError());
    return IT_OK;
  };
  auto read_totals = [&]() -> it_status {
    IT_CUDA_TRY(cudaMemcpyAsync(h, p.totals, sizeof(h), cudaMemcpyDeviceToHost, st));
    IT_CUDA_TRY(cudaStreamSynchronize(st));
    return IT_OK;
  };
  if (count_first) {
    IT_TRY(reserve(g, carve_split(p, nullptr, 0, 0, 0)));
    carve_split(p, g->slab, 0, 0, 0);
    IT_TRY(count());
    IT_TRY(read_totals());
    R = h[p.B.nb]; L = h[p.B.nb + 2]; P = h[p.B.nb + 3];
    if (R > (int64_t)INT32_MAX - 1) {
      it_set_error("split produces %lld shadow rows; row ids are 32-bit", (long long)R);
      return IT_ERR_UNSUPPORTED;
    }
  }
  IT_TRY(reserve(g, carve_split(p, nullptr, R, L, P)));
  carve_split(p, g->slab, R, L, P);
  IT_TRY(count());
  if (n > 0) {
    IT_LAUNCH(IT_K_BUCKET_SCAN, 0, 0, st, split_emit_kernel<<<split_blocks, SPLIT_THREADS, 0, st>>>(p));
    if (L > 0) {
      const int64_t cap = (int64_t)g->num_sms * 8;
      const unsigned blocks = (unsigned)(L < cap ? L : cap);
      IT_LAUNCH(IT_K_SPLIT_FILL, 0, 0, st, long_rows_kernel<<<blocks, PIECE_BINS, 0, st>>>(p));
      IT_LAUNCH(IT_K_SPLIT_FILL, 0, 0, st, long_pieces_kernel<<<blocks, PIECE_BINS, 0, st>>>(p));
    }
  } else {
    IT_CUDA_TRY(cudaMemsetAsync(g->slab, 0, g->slab_bytes, st));
  }
  IT_CUDA_TRY(cudaGetLastError());
  IT_TRY(read_totals());
  const int nb = p.B.nb;
  if (h[nb + 3] > (int64_t)INT32_MAX - 1) {
    it_set_error("%lld pieces of long vertices; they are numbered with 31 bits", (long long)h[nb + 3]);
    return IT_ERR_UNSUPPORTED;
  }
  g->shadow_indptr = p.shadow_indptr; g->shadow_owner = p.shadow_owner; g->owner_indptr = p.owner_indptr;
  g->bucket_offsets = p.bucket_offsets; g->bucket_rows = p.bucket_rows; g->list_meta = p.list_meta; g->list_owner = p.list_owner;
  g->long_owners = p.long_owners; g->piece_ptr = p.piece_ptr; g->piece_long = p.piece_long;
  g->n_rows = h[nb];
  g->n_split_owners = h[nb + 1];
  g->n_long = h[nb + 2];
  g->n_partial_rows = h[nb + 3];
  g->n_buckets = nb;
  g->n_lists = N_LISTS + 1;
  g->h_list_offsets[0] = 0;
  for (int k = 0; k < N_LISTS; ++k) {
    g->h_list_offsets[k + 1] = g->h_list_offsets[k] + h[nb + 4 + k];
    g->h_list_edges[k] = h[SPLIT_COLS + k];
    g->list_bounds[k] = k < N_FIXED && kFixedBounds[k] < p.long_above ? kFixedBounds[k] : p.long_above;   // whole vertices have no more edges
  }
  g->h_list_offsets[N_LISTS + 1] = n + (g->n_partial_rows - g->n_long);
  g->h_list_edges[N_LISTS] = h[SPLIT_COLS + IT_MAX_BUCKETS - 1];
  g->list_bounds[N_LISTS] = p.piece_max;
  for (int i = 0; i < IT_MAX_BUCKETS; ++i) g->bucket_bounds[i] = i < p.B.nb ? p.B.b[i] : 0;
  return IT_OK;
}

extern "C" it_status it_graph_set_edge_features(it_graph *g, const void *edge_feat, int32_t edge_dim, it_dtype dtype) {
  IT_REQUIRE(g != nullptr, IT_ERR_INVALID_ARG, "graph is NULL");
  if (edge_feat == nullptr || edge_dim == 0) {
    IT_REQUIRE(edge_feat == nullptr && edge_dim == 0, IT_ERR_INVALID_ARG, "edge features need both a pointer and a dimension");
    g->edge_feat = nullptr; g->edge_dim = 0;
    return IT_OK;
  }
  IT_REQUIRE(dtype == IT_F32 || dtype == IT_BF16, IT_ERR_INVALID_ARG, "bad edge feature dtype");
  const int64_t row = (int64_t)edge_dim * it_dtype_size(dtype);
  IT_REQUIRE(edge_dim > 0 && row % 16 == 0, IT_ERR_INVALID_ARG, "an edge-feature row must be a multiple of 16 bytes (got %lld)", (long long)row);
  IT_REQUIRE(((uintptr_t)edge_feat % 16) == 0, IT_ERR_INVALID_ARG, "edge features must be 16-byte aligned");
  g->edge_feat = edge_feat; g->edge_dim = edge_dim; g->edge_dtype = dtype;
  return IT_OK;
}

static it_status create_impl(int64_t n, int64_t n_src, int64_t e, const void *indptr, it_itype indptr_type,
                             const int32_t *indices, const float *edge_weights, void *stream, it_graph **out) {
  IT_REQUIRE(out != nullptr, IT_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  IT_REQUIRE(n >= 0 && n <= (int64_t)INT32_MAX - 1, IT_ERR_INVALID_ARG, "n_vertices %lld outside [0, 2^31-2]", (long long)n);
  IT_REQUIRE(n_src >= 0 && n_src <= (int64_t)INT32_MAX - 1, IT_ERR_INVALID_ARG, "n_sources %lld outside [0, 2^31-2]", (long long)n_src);
  IT_REQUIRE(e == 0 || n_src > 0, IT_ERR_INVALID_ARG, "edges need at least one source vertex");
  IT_REQUIRE(e >= 0, IT_ERR_INVALID_ARG, "n_edges is negative");
  IT_REQUIRE(indptr != nullptr, IT_ERR_INVALID_ARG, "indptr is NULL");
  IT_REQUIRE(indices != nullptr || e == 0, IT_ERR_INVALID_ARG, "indices is NULL");
  IT_REQUIRE(indptr_type == IT_I32 || indptr_type == IT_I64, IT_ERR_INVALID_ARG, "bad indptr_type");
  IT_REQUIRE(indptr_type == IT_I64 || e <= (int64_t)INT32_MAX, IT_ERR_INVALID_ARG, "int32 indptr cannot index %lld edges", (long long)e);
  cudaStream_t st = (cudaStream_t)stream;

  // one word: the validation's flags, and later the status of the graph's kernels
  int *d_status = nullptr, device = -1;
  IT_CUDA_TRY(cudaGetDevice(&device));
  IT_TRY(status_take(device, &d_status));
  IndptrView ip{indptr, indptr_type == IT_I64};
  cudaError_t ce = cudaMemsetAsync(d_status, 0, sizeof(int), st);
  int h_flags = 0;
  if (ce == cudaSuccess) {
    IT_LAUNCH(IT_K_VALIDATE, 0, 0, st, validate_indptr_kernel<<<(unsigned)((n + 1 + 255) / 256), 256, 0, st>>>(ip, n, e, d_status));
    if (e > 0) {
      const int64_t want = (e / 4 + 255) / 256, cap = (int64_t)IT_NUM_SMS_FALLBACK * 8;
      int head = (int)(((16 - ((uintptr_t)indices & 15)) & 15) / 4);
      if (head > e) head = (int)e;
      IT_LAUNCH(IT_K_VALIDATE, 0, 0, st, validate_indices_kernel<<<(unsigned)(want < 1 ? 1 : (want < cap ? want : cap)), 256, 0, st>>>(indices, e, n_src, head, d_status));
    }
    ce = cudaGetLastError();
  }
  // While the device looks the graph over: the handle, and the room for its first split (0.34 ms of the host's time; what fails here is
  // reported below, after what the graph itself may be refused for)
  it_graph *g = ce == cudaSuccess ? new (std::nothrow) it_graph() : nullptr;
  it_status room = IT_OK;
  if (g != nullptr) {
    g->n = n; g->n_src = n_src; g->e = e; g->indptr = indptr; g->indptr_type = indptr_type;
    g->indices = indices; g->edge_weights = edge_weights;
    g->device = device;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device) == cudaSuccess && sms > 0) g->num_sms = sms;
    SplitPlan plan;
    plan_split(g, 0, plan);
    if (!plan.count_first) room = reserve(g, carve_split(plan.p, nullptr, plan.R, plan.L, plan.P));
  }
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(&h_flags, d_status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
  if (ce != cudaSuccess || h_flags != 0 || g == nullptr || room != IT_OK) {
    const bool quiet = ce == cudaSuccess || cudaStreamSynchronize(st) == cudaSuccess;
    if (g != nullptr) slab_free(g);
    delete g;
    status_give_back(device, d_status, quiet);
  }
  if (ce != cudaSuccess) {
    cudaGetLastError();   // (reported here, and by no later call)
    it_set_error("graph validation failed to run: %s", cudaGetErrorString(ce));
    return IT_ERR_CUDA;
  }
  if (h_flags != 0) {
    it_set_error("bad CSR:%s%s%s%s", (h_flags & 1) ? " indptr[0] != 0;" : "", (h_flags & 2) ? " indptr decreases;" : "",
                 (h_flags & 4) ? " indptr[n] != n_edges;" : "", (h_flags & 8) ? " a source id is outside [0, n_sources);" : "");
    return IT_ERR_BAD_GRAPH;
  }
  if (room != IT_OK) return room;   // (its text is set)
  IT_REQUIRE(g != nullptr, IT_ERR_OOM, "host allocation failed");
  g->d_status = d_status;   // zero: the flags were
  it_status rc = split_impl(g, 0, st);
  if (rc != IT_OK) { it_graph_destroy(g); return rc; }
  *out = g;
  return IT_OK;
}

extern "C" it_status it_graph_create(int64_t n, int64_t e, const void *indptr, it_itype indptr_type,
                                     const int32_t *indices, const float *edge_weights, void *stream,
                                     it_graph **out) {
  return create_impl(n, n, e, indptr, indptr_type, indices, edge_weights, stream, out);
}

extern "C" it_status it_graph_create_part(int64_t n, int64_t n_sources, int64_t e, const void *indptr, it_itype indptr_type,
                                          const int32_t *indices, const float *edge_weights, void *stream,
                                          it_graph **out) {
  return create_impl(n, n_sources, e, indptr, indptr_type, indices, edge_weights, stream, out);
}

extern "C" it_status it_split_hubs(it_graph *g, int64_t threshold, void *stream, int64_t *out_n_rows,
                                   int64_t *out_n_split_owners) {
  IT_REQUIRE(g != nullptr, IT_ERR_INVALID_ARG, "graph is NULL");
  IT_TRY(split_impl(g, threshold, (cudaStream_t)stream));
  if (out_n_rows) *out_n_rows = g->n_rows;
  if (out_n_split_owners) *out_n_split_owners = g->n_split_owners;
  return IT_OK;
}

extern "C" it_status it_graph_get_split(const it_graph *g, int64_t *n_rows, const int64_t **shadow_indptr,
                                        const int32_t **shadow_owner, const int64_t **owner_indptr,
                                        const int64_t **bucket_offsets, const int32_t **bucket_rows,
                                        int32_t *n_buckets, int64_t *bucket_bounds) {
  IT_REQUIRE(g != nullptr, IT_ERR_INVALID_ARG, "graph is NULL");
  g->used = true;
  if (n_rows) *n_rows = g->n_rows;
  if (shadow_indptr) *shadow_indptr = g->shadow_indptr;
  if (shadow_owner) *shadow_owner = g->shadow_owner;
  if (owner_indptr) *owner_indptr = g->owner_indptr;
  if (bucket_offsets) *bucket_offsets = g->bucket_offsets;
  if (bucket_rows) *bucket_rows = g->bucket_rows;
  if (n_buckets) *n_buckets = g->n_buckets;
  if (bucket_bounds) memcpy(bucket_bounds, g->bucket_bounds, sizeof(g->bucket_bounds));
  return IT_OK;
}

extern "C" it_status it_graph_check(it_graph *g, void *stream) {
  IT_REQUIRE(g != nullptr, IT_ERR_INVALID_ARG, "graph is NULL");
  cudaStream_t st = (cudaStream_t)stream;
  int h = 0;
  IT_CUDA_TRY(cudaMemcpyAsync(&h, g->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
  IT_CUDA_TRY(cudaStreamSynchronize(st));
  if (h != 0) {
    IT_CUDA_TRY(cudaMemsetAsync(g->d_status, 0, sizeof(int), st));
    it_set_error("a kernel gave up a bounded wait; its outputs are not valid");
    return IT_ERR_TIMEOUT;
  }
  return IT_OK;
}

extern "C" it_status it_graph_destroy(it_graph *g) {
  if (!g) return IT_OK;
  const bool quiet = g->slab != nullptr;   // (its release waits)
  slab_free(g);
  status_give_back(g->device, g->d_status, quiet);
  delete g;
  return IT_OK;
}
