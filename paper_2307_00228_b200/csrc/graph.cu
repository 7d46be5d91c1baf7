// Graph ingest, validation, hub split into shadow rows, degree buckets.
// Integer-only work; every array produced here is a pure function of (indptr, threshold)
// and is built without atomics on data, so it is reproducible bit for bit.
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
__global__ void __launch_bounds__(256) validate_indices_kernel(const int32_t *__restrict__ idx, int64_t e, int64_t n, int head, int *flags) {
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
// numbers, the list of split vertices and the positions inside every bucket are prefix sums of the same pass: columns
// 0 .. nb - 1 the buckets, nb the rows, nb + 1 the split vertices.
// Bound by reading indptr twice and writing 36 bytes per row; a scan per bucket (each over every row, three launches with a
// read of two 8-byte bounds per row) took 3.2 ms of device time for 5M vertices and six buckets, this one 3.0 with
// everything around it (create + split: 14.3 -> 3.0 ms; the derived arrays are one allocation instead of nine, kept for the next split).
constexpr int SPLIT_THREADS = 256;
constexpr int SPLIT_ITEMS = 8;                                    // vertices per lane: a warp covers 256 consecutive ones
constexpr int SPLIT_TILE = SPLIT_THREADS * SPLIT_ITEMS;
constexpr int SPLIT_COLS = IT_MAX_BUCKETS + 2;

struct Bounds { int64_t b[IT_MAX_BUCKETS]; int nb; };
__device__ __forceinline__ int bucket_of(int64_t len, const Bounds &B) {
  int k = 0;
  while (k < B.nb - 1 && len > B.b[k]) ++k;
  return k;
}

struct SplitInfo { int64_t r0, pos_a, pos_b; };   // a split vertex: its first row; list positions of its longer / shorter groups

struct SplitParams {
  IndptrView ip;
  int64_t n, e, T;
  Bounds B;
  int64_t n_tiles;
  int64_t *tiles;          // [SPLIT_COLS][n_tiles]
  int64_t *totals;         // [SPLIT_COLS] column sums, then [IT_MAX_BUCKETS] edges per bucket
  int64_t *shadow_indptr; int32_t *shadow_owner; int64_t *owner_indptr; int32_t *split_owners;
  int64_t *bucket_offsets; int32_t *bucket_rows; it_row_meta *bucket_meta; int32_t *bucket_owner;
  SplitInfo *info;         // [split vertices]
};

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

// Lane c of a warp keeps column c.  One step over 32 vertices, of which those in `valid` exist: count(...) adds them.
__device__ __forceinline__ void add_columns(int64_t &col, const VertexRows &r, unsigned valid, unsigned split, int nb, int lane) {
  const bool plain = ((valid & ~split) >> lane) & 1u;
  for (int k = 0; k < nb; ++k) {
    const unsigned m = __ballot_sync(0xffffffffu, plain && r.ka == k);
    if (lane == k) col += __popc(m);
  }
  if (lane == nb) col += __popc(valid & ~split);
  while (split) {   // rare
    const int l = __ffs(split) - 1;
    split &= split - 1;
    const int64_t ng = __shfl_sync(0xffffffffu, r.ng, l), rem = __shfl_sync(0xffffffffu, r.rem, l);
    const int ka = __shfl_sync(0xffffffffu, r.ka, l), kb = __shfl_sync(0xffffffffu, r.kb, l);
    if (lane == ka) col += rem;
    if (lane == kb) col += ng - rem;
    if (lane == nb) col += ng;
    if (lane == nb + 1) col += 1;
  }
}

__global__ void __launch_bounds__(SPLIT_THREADS) split_count_kernel(SplitParams p) {
  __shared__ unsigned long long cols[SPLIT_COLS], edges[IT_MAX_BUCKETS];
  const int lane = threadIdx.x & 31, nb = p.B.nb;
  if (threadIdx.x < SPLIT_COLS) cols[threadIdx.x] = 0;
  if (threadIdx.x < IT_MAX_BUCKETS) edges[threadIdx.x] = 0;
  __syncthreads();
  const int64_t v0 = (int64_t)blockIdx.x * SPLIT_TILE + (int64_t)(threadIdx.x >> 5) * (32 * SPLIT_ITEMS) + lane;
  int64_t col = 0, my_edges = 0;
  for (int i = 0; i < SPLIT_ITEMS; ++i) {
    const int64_t v = v0 + i * 32;
    const int64_t d = v < p.n ? p.ip[v + 1] - p.ip[v] : 0;
    const VertexRows r = rows_of(d, p);
    const unsigned valid = __ballot_sync(0xffffffffu, v < p.n), split = __ballot_sync(0xffffffffu, r.ng > 1);
    if (valid == 0) break;
    add_columns(col, r, valid, split, nb, lane);
    // edges per bucket: 32-bit sums across the lanes unless a vertex is huge
    if (__any_sync(0xffffffffu, d >= ((int64_t)1 << 26) || r.ng > 1)) {
      if (v < p.n) {
        const int64_t in_a = r.rem * (r.ng > 1 ? d / r.ng + 1 : 0);
        if (in_a) atomicAdd(&edges[r.ka], (unsigned long long)in_a);
        atomicAdd(&edges[r.kb], (unsigned long long)(d - in_a));
      }
    } else {
      for (int k = 0; k < nb; ++k) {
        const unsigned s = __reduce_add_sync(0xffffffffu, r.kb == k ? (unsigned)d : 0u);
        if (lane == k) my_edges += s;
      }
    }
  }
  if (lane < nb + 2) atomicAdd(&cols[lane], (unsigned long long)col);
  if (lane < nb) atomicAdd(&edges[lane], (unsigned long long)my_edges);
  __syncthreads();
  if (threadIdx.x < nb + 2) p.tiles[threadIdx.x * p.n_tiles + blockIdx.x] = (int64_t)cols[threadIdx.x];
  if (threadIdx.x < nb && edges[threadIdx.x])
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
  __shared__ int64_t warp_cols[SPLIT_THREADS / 32][SPLIT_COLS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nb = p.B.nb;
  const int64_t v0 = (int64_t)blockIdx.x * SPLIT_TILE + (int64_t)warp * (32 * SPLIT_ITEMS) + lane;
  int64_t j0[SPLIT_ITEMS];
  int64_t d[SPLIT_ITEMS];
  int64_t col = 0;
#pragma unroll
  for (int i = 0; i < SPLIT_ITEMS; ++i) {
    const int64_t v = v0 + i * 32;
    j0[i] = v < p.n ? p.ip[v] : 0;
    d[i] = v < p.n ? p.ip[v + 1] - j0[i] : 0;
    const VertexRows r = rows_of(d[i], p);
    add_columns(col, r, __ballot_sync(0xffffffffu, v < p.n), __ballot_sync(0xffffffffu, r.ng > 1), nb, lane);
  }
  if (lane < nb + 2) warp_cols[warp][lane] = col;
  __syncthreads();
  // lane c: the running value of column c; for a bucket counted from the start of the whole list
  int64_t run = 0;
  if (lane < nb + 2) {
    run = p.tiles[lane * p.n_tiles + blockIdx.x];
    for (int w = 0; w < warp; ++w) run += warp_cols[w][lane];
    if (lane < nb)
      for (int k = 0; k < lane; ++k) run += p.totals[k];
  }
  if (blockIdx.x == 0 && warp == 0) {
    if (lane <= nb) {
      int64_t off = 0;
      for (int k = 0; k < lane; ++k) off += p.totals[k];
      p.bucket_offsets[lane] = off;
    }
    if (lane == 0) {
      p.shadow_indptr[p.totals[nb]] = p.e;
      p.owner_indptr[p.n] = p.totals[nb];
    }
  }
#pragma unroll
  for (int i = 0; i < SPLIT_ITEMS; ++i) {
    const int64_t v = v0 + i * 32;
    const VertexRows r = rows_of(d[i], p);
    const unsigned valid = __ballot_sync(0xffffffffu, v < p.n), split = __ballot_sync(0xffffffffu, r.ng > 1);
    int64_t row = 0, pos = 0;
    if (split == 0) {
      row = __shfl_sync(0xffffffffu, run, nb) + lane;
      for (int k = 0; k < nb; ++k) {
        const unsigned m = __ballot_sync(0xffffffffu, v < p.n && r.ka == k);
        const int64_t at = __shfl_sync(0xffffffffu, run, k);
        if (r.ka == k) pos = at + __popc(m & ((1u << lane) - 1u));
      }
      add_columns(run, r, valid, 0u, nb, lane);
    } else {   // a split vertex among the 32: one vertex after the other
      for (int l = 0; l < 32; ++l) {
        if (!((valid >> l) & 1u)) break;
        const int64_t ng = __shfl_sync(0xffffffffu, r.ng, l), rem = __shfl_sync(0xffffffffu, r.rem, l);
        const int ka = __shfl_sync(0xffffffffu, r.ka, l), kb = __shfl_sync(0xffffffffu, r.kb, l);
        const int64_t at_row = __shfl_sync(0xffffffffu, run, nb), at_k = __shfl_sync(0xffffffffu, run, nb + 1);
        if (lane == nb) run += ng;
        if (lane == nb + 1 && ng > 1) run += 1;
        const int64_t at_a = __shfl_sync(0xffffffffu, run, ka);
        if (ng > 1 && lane == ka) run += rem;
        const int64_t at_b = __shfl_sync(0xffffffffu, run, kb);
        if (lane == kb) run += ng - rem;   // (one plain row: rem = 0)
        if (lane == l) {
          row = at_row; pos = at_b;
          if (ng > 1) {
            p.split_owners[at_k] = (int32_t)v;
            p.info[at_k] = SplitInfo{at_row, at_a, at_b};
          }
        }
      }
    }
    if (v < p.n) {
      p.owner_indptr[v] = row;
      if (r.ng == 1) {
        p.shadow_indptr[row] = j0[i];
        p.shadow_owner[row] = (int32_t)v;
        p.bucket_rows[pos] = (int32_t)row;
        it_row_meta m;
        m.j0 = j0[i]; m.len = (int32_t)d[i]; m.dest = (int32_t)v;
        p.bucket_meta[pos] = m;
        p.bucket_owner[pos] = (int32_t)v;
      }
    }
  }
}

// Rows of split vertices: one block per split vertex, groups written by closed form
//   start(g) = indptr[v] + g * base + min(g, rem),  base = d / ng, rem = d % ng;
// group g's partial result goes to slot p0 + g: the rows of earlier split vertices = all earlier rows minus earlier unsplit vertices.
__global__ void __launch_bounds__(128) fill_split_rows_kernel(SplitParams p) {
  const int64_t n_split = p.totals[p.B.nb + 1];
  for (int64_t k = blockIdx.x; k < n_split; k += gridDim.x) {
    const int64_t v = p.split_owners[k], s = p.ip[v], d = p.ip[v + 1] - s;
    const SplitInfo f = p.info[k];
    const int64_t ng = groups_of(d, p.T), base = d / ng, rem = d % ng, p0 = f.r0 - v + k;
    for (int64_t g = threadIdx.x; g < ng; g += blockDim.x) {
      const int64_t row = f.r0 + g, pos = g < rem ? f.pos_a + g : f.pos_b + (g - rem);
      it_row_meta m;
      m.j0 = s + g * base + (g < rem ? g : rem);
      m.len = (int32_t)(base + (g < rem ? 1 : 0));
      m.dest = (int32_t)~(p0 + g);
      p.shadow_indptr[row] = m.j0;
      p.shadow_owner[row] = (int32_t)v;
      p.bucket_rows[pos] = (int32_t)row;
      p.bucket_meta[pos] = m;
      p.bucket_owner[pos] = (int32_t)v;
    }
  }
}

// ----------------------------------------------------------------------------- host side
static void forget_split(it_graph *g) {
  g->shadow_indptr = nullptr; g->shadow_owner = nullptr; g->owner_indptr = nullptr;
  g->split_owners = nullptr; g->bucket_offsets = nullptr; g->bucket_rows = nullptr;
  g->bucket_meta = nullptr; g->bucket_owner = nullptr;
  g->n_rows = g->n_split_owners = g->n_partial_rows = 0;
  g->n_buckets = 0;
}

// The derived arrays and the scratch of a split with at most R rows and S split vertices, carved out of one allocation that
// the graph keeps for its next split (NULL slab: only the size).
static size_t carve_split(it_graph *g, SplitParams &p, char *slab, int64_t R, int64_t S) {
  size_t off = 0;
  auto take = [&](auto *&ptr, int64_t count) {
    ptr = reinterpret_cast<std::remove_reference_t<decltype(ptr)>>(slab + off);
    off += it_align_up((size_t)(count > 0 ? count : 1) * sizeof(*ptr));
  };
  take(p.totals, SPLIT_COLS + IT_MAX_BUCKETS);
  take(p.tiles, SPLIT_COLS * p.n_tiles);
  take(p.bucket_offsets, IT_MAX_BUCKETS + 1);
  take(p.owner_indptr, p.n + 1);
  take(p.shadow_indptr, R + 1);
  take(p.shadow_owner, R);
  take(p.bucket_rows, R);
  take(p.bucket_meta, R);
  take(p.bucket_owner, R);
  take(p.split_owners, S);
  take(p.info, S);
  return off;
}

static it_status split_impl(it_graph *g, int64_t T, cudaStream_t st) {
  // the arrays of the previous split are written over: forward passes on any stream that still read them come first
  if (g->bucket_meta) IT_CUDA_TRY(cudaDeviceSynchronize());
  forget_split(g);
  g->threshold = T > 0 ? T : 0;
  const int64_t n = g->n;
  SplitParams p{};
  p.ip = IndptrView{g->indptr, g->indptr_type == IT_I64};
  p.n = n; p.e = g->e; p.T = T;
  p.n_tiles = (n + SPLIT_TILE - 1) / SPLIT_TILE;
  // degree buckets: {0, 8, 32, 256, 1024, everything longer}
  const int64_t fixed[5] = {0, 8, 32, 256, 1024};
  p.B.nb = 0;
  for (int i = 0; i < 5; ++i)
    if (T <= 0 || fixed[i] < T) p.B.b[p.B.nb++] = fixed[i];
  p.B.b[p.B.nb++] = T > 0 ? T : INT64_MAX;

  // at most one row per vertex and one more per T edges; only where that is far above the number of vertices are the rows
  // counted before the arrays are laid out
  int64_t R = n + (T > 0 ? g->e / T : 0), S = T > 0 ? (n < g->e / T ? n : g->e / T) : 0;
  const bool count_first = R > n + n / 4 + (1 << 20) || R > (int64_t)INT32_MAX - 1;
  int64_t h[SPLIT_COLS + IT_MAX_BUCKETS] = {0};
  auto reserve = [&](size_t bytes) -> it_status {   // grow the graph's allocation; what it holds is not kept
    if (bytes <= g->slab_bytes) return IT_OK;
    cudaFree(g->slab);
    g->slab = nullptr; g->slab_bytes = 0;
    IT_CUDA_TRY(cudaMalloc(&g->slab, bytes));
    g->slab_bytes = bytes;
    return IT_OK;
  };
  auto count = [&]() -> it_status {
    IT_CUDA_TRY(cudaMemsetAsync(p.totals, 0, sizeof(h), st));
    if (n > 0) {
      IT_LAUNCH(IT_K_SPLIT_SCAN, 0, 0, st, split_count_kernel<<<(unsigned)p.n_tiles, SPLIT_THREADS, 0, st>>>(p));
      IT_LAUNCH(IT_K_SPLIT_SCAN, 0, 0, st, split_scan_kernel<<<(unsigned)(p.B.nb + 2), 1024, 0, st>>>(p));
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
    IT_TRY(reserve(carve_split(g, p, nullptr, 0, 0)));
    carve_split(g, p, g->slab, 0, 0);
    IT_TRY(count());
    IT_TRY(read_totals());
    R = h[p.B.nb]; S = h[p.B.nb + 1];
    if (R > (int64_t)INT32_MAX - 1) {
      it_set_error("split produces %lld shadow rows; row ids are 32-bit", (long long)R);
      return IT_ERR_UNSUPPORTED;
    }
  }
  IT_TRY(reserve(carve_split(g, p, nullptr, R, S)));
  carve_split(g, p, g->slab, R, S);
  IT_TRY(count());
  if (n > 0) {
    IT_LAUNCH(IT_K_BUCKET_SCAN, 0, 0, st, split_emit_kernel<<<(unsigned)p.n_tiles, SPLIT_THREADS, 0, st>>>(p));
    if (S > 0) {
      const int64_t cap = (int64_t)g->num_sms * 16;
      IT_LAUNCH(IT_K_SPLIT_FILL, 0, 0, st, fill_split_rows_kernel<<<(unsigned)(S < cap ? S : cap), 128, 0, st>>>(p));
    }
  } else {
    IT_CUDA_TRY(cudaMemsetAsync(g->slab, 0, g->slab_bytes, st));
  }
  IT_CUDA_TRY(cudaGetLastError());
  IT_TRY(read_totals());
  g->shadow_indptr = p.shadow_indptr; g->shadow_owner = p.shadow_owner; g->owner_indptr = p.owner_indptr; g->split_owners = p.split_owners;
  g->bucket_offsets = p.bucket_offsets; g->bucket_rows = p.bucket_rows; g->bucket_meta = p.bucket_meta; g->bucket_owner = p.bucket_owner;
  g->n_rows = h[p.B.nb];
  g->n_split_owners = h[p.B.nb + 1];
  g->n_partial_rows = g->n_rows - (n - g->n_split_owners);
  g->n_buckets = p.B.nb;
  g->h_bucket_offsets[0] = 0;
  for (int k = 0; k < p.B.nb; ++k) {
    g->h_bucket_offsets[k + 1] = g->h_bucket_offsets[k] + h[k];
    g->h_bucket_edges[k] = h[SPLIT_COLS + k];
  }
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
  int *d_status = nullptr;
  IT_CUDA_TRY(cudaMalloc(&d_status, sizeof(int)));
  IndptrView ip{indptr, indptr_type == IT_I64};
  cudaError_t ce = cudaMemsetAsync(d_status, 0, sizeof(int), st);
  int h_flags = 0;
  if (ce == cudaSuccess) {
    IT_LAUNCH(IT_K_VALIDATE, 0, 0, st, validate_indptr_kernel<<<(unsigned)((n + 1 + 255) / 256), 256, 0, st>>>(ip, n, e, d_status));
    if (e > 0) {   // the caller vouches for e source ids, whatever indptr says
      const int64_t want = (e / 4 + 255) / 256, cap = (int64_t)IT_NUM_SMS_FALLBACK * 8;
      int head = (int)(((16 - ((uintptr_t)indices & 15)) & 15) / 4);
      if (head > e) head = (int)e;
      IT_LAUNCH(IT_K_VALIDATE, 0, 0, st, validate_indices_kernel<<<(unsigned)(want < 1 ? 1 : (want < cap ? want : cap)), 256, 0, st>>>(indices, e, n_src, head, d_status));
    }
    ce = cudaGetLastError();
  }
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(&h_flags, d_status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
  if (ce != cudaSuccess || h_flags != 0) cudaFree(d_status);
  if (ce != cudaSuccess) {
    it_set_error("graph validation failed to run: %s", cudaGetErrorString(ce));
    return IT_ERR_CUDA;
  }
  if (h_flags != 0) {
    it_set_error("bad CSR:%s%s%s%s", (h_flags & 1) ? " indptr[0] != 0;" : "", (h_flags & 2) ? " indptr decreases;" : "",
                 (h_flags & 4) ? " indptr[n] != n_edges;" : "", (h_flags & 8) ? " a source id is outside [0, n_sources);" : "");
    return IT_ERR_BAD_GRAPH;
  }

  it_graph *g = new (std::nothrow) it_graph();
  if (g == nullptr) cudaFree(d_status);
  IT_REQUIRE(g != nullptr, IT_ERR_OOM, "host allocation failed");
  g->n = n; g->n_src = n_src; g->e = e; g->indptr = indptr; g->indptr_type = indptr_type;
  g->indices = indices; g->edge_weights = edge_weights;
  g->d_status = d_status;   // zero: the flags were
  cudaGetDevice(&g->device);
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, g->device) == cudaSuccess && sms > 0) g->num_sms = sms;
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
  cudaFree(g->slab);
  cudaFree(g->d_status);
  delete g;
  return IT_OK;
}
