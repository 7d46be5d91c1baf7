// Gather and combine: the column chunks of a row go to the kernels of gather_rows.cuh; the partial results of a split
// vertex are folded here.
#include "stream.cuh"

it_status it_launch_gather_rows_f32(const it_gather_args &a, const it_stream::StreamParams &sp, bool *folded, cudaStream_t st);
it_status it_launch_gather_rows_bf16(const it_gather_args &a, const it_stream::StreamParams &sp, bool *folded, cudaStream_t st);

namespace {

using namespace it_stream;
constexpr int GATHER_THREADS = THREADS;
constexpr int64_t EDGE_RUN = 512;

// ----------------------------------------------------------------------------- combine
// One block per long vertex.  Its partial rows are rows [piece_ptr[k], piece_ptr[k + 1]) of the partial buffer; every warp
// folds a contiguous range of them in order, eight rows in flight, and the warps' results are folded in warp order.
// EDGES: where there is no partial buffer (a layer that just fits the built-in scratch) the same is done over the source rows of
// the vertex's edges.
struct CombineParams {
  const int32_t *__restrict__ long_owners;
  const int64_t *__restrict__ piece_ptr;
  const int64_t *__restrict__ owner_indptr;
  const int64_t *__restrict__ shadow_indptr;
  const float *__restrict__ partials;
  const char *__restrict__ src;          // EDGES: rows of T, src_pitch bytes from one to the next, ...
  const int32_t *__restrict__ indices;   // ... by source vertex (NULL: by edge), ...
  const float *__restrict__ weights;     // ... and their weights (NULL: 1)
  void *__restrict__ dst;
  const void *__restrict__ self_term;
  const float *__restrict__ bias;
  int64_t n_long, src_pitch;
  int dim, dst_ld, self_ld;
  int red, is_mean, epi, act;   // red: RED_SUM / RED_MAX / RED_MIN
};

template <typename T, bool EDGES>
__global__ void __launch_bounds__(GATHER_THREADS) combine_kernel(CombineParams p) {
  constexpr int WARPS = GATHER_THREADS / 32;
  __shared__ float4 red[WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t k = blockIdx.x; k < p.n_long; k += gridDim.x) {
    const int64_t v = __ldg(p.long_owners + k);
    const int64_t j0 = __ldg(p.shadow_indptr + __ldg(p.owner_indptr + v)), deg = __ldg(p.shadow_indptr + __ldg(p.owner_indptr + v + 1)) - j0;
    const int64_t p0 = EDGES ? j0 : __ldg(p.piece_ptr + k), n = EDGES ? deg : __ldg(p.piece_ptr + k + 1) - p0;
    const int64_t per = (n + WARPS - 1) / WARPS;
    const int64_t a = warp * per < n ? warp * per : n, b = a + per < n ? a + per : n;
    for (int c0 = 0; c0 < p.dim; c0 += 128) {
      const int c = c0 + lane * 4;
      const float id = p.red == RED_MAX ? -INFINITY : (p.red == RED_MIN ? INFINITY : 0.f);
      float4 acc = make_float4(id, id, id, id);
      auto fold = [&](const float4 &y) {
        if (p.red == RED_MAX) {
          acc.x = fmaxf(acc.x, y.x); acc.y = fmaxf(acc.y, y.y); acc.z = fmaxf(acc.z, y.z); acc.w = fmaxf(acc.w, y.w);
        } else if (p.red == RED_MIN) {
          acc.x = fminf(acc.x, y.x); acc.y = fminf(acc.y, y.y); acc.z = fminf(acc.z, y.z); acc.w = fminf(acc.w, y.w);
        } else {
          acc.x += y.x; acc.y += y.y; acc.z += y.z; acc.w += y.w;
        }
      };
      if constexpr (EDGES) {
        using Slice = RowSlice<T, 4 * (int)sizeof(T)>;
        if (c < p.dim) {
          auto edge = [&](const typename Slice::Raw &raw, float w) {
            float y[4];
            Slice::unpack(raw, y);
            if (p.red == RED_SUM) { acc.x = fmaf(w, y[0], acc.x); acc.y = fmaf(w, y[1], acc.y); acc.z = fmaf(w, y[2], acc.z); acc.w = fmaf(w, y[3], acc.w); }
            else fold(make_float4(w * y[0], w * y[1], w * y[2], w * y[3]));
          };
          auto load = [&](int64_t j) { return Slice::load(p.src + (p.indices ? (int64_t)__ldg(p.indices + j) : j) * p.src_pitch + (size_t)c * sizeof(T)); };
          float4 total = acc;
          for (int64_t g = a; g < b;) {   // in runs as long as a piece, so that sums are rounded no more often than with partial rows
            const int64_t end = b - g < EDGE_RUN ? b : g + EDGE_RUN;
            acc = make_float4(id, id, id, id);
            for (; g + 8 <= end; g += 8) {
              typename Slice::Raw y[8];
#pragma unroll
              for (int u = 0; u < 8; ++u) y[u] = load(p0 + g + u);
#pragma unroll
              for (int u = 0; u < 8; ++u) edge(y[u], p.weights ? __ldg(p.weights + p0 + g + u) : 1.f);
            }
            for (; g < end; ++g) edge(load(p0 + g), p.weights ? __ldg(p.weights + p0 + g) : 1.f);
            const float4 run = acc;
            acc = total;
            fold(run);
            total = acc;
          }
        }
      } else if (c < p.dim) {
        const float *P = p.partials + p0 * p.dim + c;
        int64_t g = a;
        for (; g + 8 <= b; g += 8) {
          float4 y[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) y[u] = __ldcs(reinterpret_cast<const float4 *>(P + (g + u) * p.dim));
#pragma unroll
          for (int u = 0; u < 8; ++u) fold(y[u]);
        }
        for (; g < b; ++g) fold(__ldcs(reinterpret_cast<const float4 *>(P + g * p.dim)));
      }
      __syncthreads();   // red free again
      red[warp][lane] = acc;
      __syncthreads();
      if (warp != 0 || c >= p.dim) continue;   // (the barriers above are met by every warp in every round)
      for (int w = 1; w < WARPS; ++w) fold(red[w][lane]);
      const float inv = p.is_mean ? 1.f / (float)deg : 1.f;
      float o[4] = {acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv};
      const int64_t doff = v * p.dst_ld + c;
      if (p.epi == IT_EPI_RAW_F32) {
        *reinterpret_cast<float4 *>(reinterpret_cast<float *>(p.dst) + doff) = make_float4(o[0], o[1], o[2], o[3]);
        continue;
      }
      if (p.epi == IT_EPI_ADD_ACT) {
        float4 s;
        if constexpr (sizeof(T) == 2) {
          const uint2 raw = __ldg(reinterpret_cast<const uint2 *>(reinterpret_cast<const T *>(p.self_term) + v * p.self_ld + c));
          s = make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xffff0000u), __uint_as_float(raw.y << 16),
                          __uint_as_float(raw.y & 0xffff0000u));
        } else {
          s = __ldg(reinterpret_cast<const float4 *>(reinterpret_cast<const float *>(p.self_term) + v * p.self_ld + c));
        }
        o[0] = act_apply(o[0] + s.x, p.act); o[1] = act_apply(o[1] + s.y, p.act);
        o[2] = act_apply(o[2] + s.z, p.act); o[3] = act_apply(o[3] + s.w, p.act);
      } else if (p.epi == IT_EPI_BIAS_ACT) {
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = act_apply(o[i] + (p.bias ? __ldg(p.bias + c + i) : 0.f), p.act);
      }
      T *d = reinterpret_cast<T *>(p.dst) + doff;
      if (sizeof(T) == 4) {
        *reinterpret_cast<float4 *>(d) = make_float4(o[0], o[1], o[2], o[3]);
      } else {
        __nv_bfloat162 h0 = __floats2bfloat162_rn(o[0], o[1]), h1 = __floats2bfloat162_rn(o[2], o[3]);
        *reinterpret_cast<uint2 *>(d) = make_uint2(*reinterpret_cast<uint32_t *>(&h0), *reinterpret_cast<uint32_t *>(&h1));
      }
    }
  }
}

// ----------------------------------------------------------------------------- rows without edges
__global__ void __launch_bounds__(GATHER_THREADS) empty_rows_kernel(EmptyRowsParams p) {
  __shared__ uint4 row[128];   // rows of up to 512 entries
  if (p.kind != IT_EMPTY_SELF) {
    for (int s = threadIdx.x; s < p.slices; s += GATHER_THREADS) row[s] = empty_piece(p, s);
    __syncthreads();
  }
  for (int64_t b = p.lo + ((int64_t)blockIdx.x * (GATHER_THREADS / 32) + (threadIdx.x >> 5)) * 32; b < p.hi; b += (int64_t)gridDim.x * GATHER_THREADS)
    empty_rows_warp(p, b, (int)(p.hi - b < 32 ? p.hi - b : 32), threadIdx.x & 31, [&](int s) { return row[s]; });
}

}  // namespace

it_status it_launch_empty_rows(const it_empty_rows_args &a, int kid, double bytes, cudaStream_t st) {
  const it_graph *g = a.g;
  EmptyRowsParams p;
  p.meta = g->list_meta; p.lo = a.row_lo; p.hi = a.row_hi; p.dst = (char *)a.dst; p.pitch = a.pitch;
  p.self = (const char *)a.self; p.self_pitch = a.self_pitch; p.kind = (int)a.kind;
  p.slices = a.dim * it_dtype_size(a.dtype) / 16; p.bf16 = a.dtype == IT_BF16; p.act = (int)a.act;
  p.value = a.value; p.bias = a.bias;
  const int64_t want = (a.row_hi - a.row_lo + GATHER_THREADS - 1) / GATHER_THREADS, cap = (int64_t)g->num_sms * 8;
  IT_LAUNCH(kid, bytes, 0, st, empty_rows_kernel<<<(unsigned)(want < cap ? want : cap), GATHER_THREADS, 0, st>>>(p));
  IT_CUDA_TRY(cudaGetLastError());
  return IT_OK;
}

// One column chunk of the rows: `a.dim` is the chunk's width (16 to 512 bytes), the
// pointers already point at its first column, and the *_ld fields / src_ld carry the full row lengths.
static it_status launch_gather_chunk(const it_gather_args &a, cudaStream_t st) {
  const it_graph *g = a.g;
  bool folded = false;   // the pieces of long vertices, by the kernel that walked them
  StreamParams sp;
  sp.meta = g->list_meta; sp.owner = nullptr; sp.indices = a.per_edge_rows ? nullptr : g->indices; sp.weights = g->edge_weights;
  sp.src = a.src; sp.row_lo = sp.row_hi = 0; sp.dim = a.dim; sp.batch_rows = 1; sp.counter = nullptr; sp.claim = 1; sp.slices = 0;
  sp.src_pitch = (uint32_t)((a.src_ld > 0 ? a.src_ld : a.dim) * it_dtype_size(a.dtype));
  if (a.dtype == IT_F32) IT_TRY(it_launch_gather_rows_f32(a, sp, &folded, st));
  else IT_TRY(it_launch_gather_rows_bf16(a, sp, &folded, st));
  if (g->n_long > 0 && !folded) {
    CombineParams c;
    c.long_owners = g->long_owners; c.piece_ptr = g->piece_ptr; c.owner_indptr = g->owner_indptr; c.shadow_indptr = g->shadow_indptr;
    c.partials = a.partials; c.src = (const char *)a.src; c.src_pitch = sp.src_pitch; c.indices = sp.indices; c.weights = a.use_edge_weights ? g->edge_weights : nullptr;
    c.dst = a.dst; c.self_term = a.self_term; c.bias = a.bias; c.n_long = g->n_long;
    c.dim = a.dim; c.dst_ld = a.dst_ld > 0 ? a.dst_ld : a.dim; c.self_ld = a.self_ld > 0 ? a.self_ld : a.dim;
    c.red = a.op == IT_GATHER_MAX ? RED_MAX : (a.op == IT_GATHER_MIN ? RED_MIN : RED_SUM); c.is_mean = a.op == IT_GATHER_MEAN && a.epi != IT_EPI_RAW_F32; c.epi = a.epi; c.act = a.act;
    const int64_t cap = (int64_t)g->num_sms * 8;
    const unsigned blocks = (unsigned)(g->n_long < cap ? g->n_long : cap);
    const double es = it_dtype_size(a.dtype);
    const double cbytes = (a.partials ? (double)g->n_partial_rows * a.dim * 4.0 : (double)g->h_list_edges[g->n_lists - 1] * (4.0 + a.dim * es)) + (double)g->n_long * a.dim * es;
    auto go = [&]<typename T>() {
      if (a.partials) IT_LAUNCH(IT_K_COMBINE, cbytes, 0, st, combine_kernel<T, false><<<blocks, GATHER_THREADS, 0, st>>>(c));
      else IT_LAUNCH(IT_K_COMBINE, cbytes, 0, st, combine_kernel<T, true><<<blocks, GATHER_THREADS, 0, st>>>(c));
    };
    if (a.dtype == IT_F32) go.template operator()<float>();
    else go.template operator()<__nv_bfloat16>();
    IT_CUDA_TRY(cudaGetLastError());
  }
  return IT_OK;
}

// Rows of any multiple of 16 bytes: the kernels take rows of up to 512 bytes, so a wider row is cut into column chunks and
// each chunk is gathered on its own, reading and writing
// its columns in place.  The aggregate is entry by entry, so the chunks are independent; each pass re-reads
// the edge indices (4 bytes against a chunk of up to 512 per edge).
it_status it_launch_gather(const it_gather_args &a, cudaStream_t st) {
  const it_graph *g = a.g;
  IT_REQUIRE(a.op == IT_GATHER_SUM || a.op == IT_GATHER_MEAN || a.op == IT_GATHER_MAX || a.op == IT_GATHER_MIN, IT_ERR_INVALID_ARG,
             "gather: bad op");
  IT_REQUIRE(!a.use_edge_weights || g->edge_weights, IT_ERR_INVALID_ARG, "layer uses edge weights but the graph has none");
  const int es = it_dtype_size(a.dtype);
  IT_REQUIRE(a.dim > 0 && (a.dim * es) % 16 == 0, IT_ERR_INVALID_ARG, "gather: a row of %d bytes is not a multiple of 16", a.dim * es);
  if (g->n == 0) return IT_OK;
  const int full = a.dim;
  int c0 = 0;   // first column of the chunk
  while (c0 < full) {
    const int left = (full - c0) * es;
    const int bytes = left >= 512 ? 512 : left;
    it_gather_args c = a;
    c.dim = bytes / es;
    c.src = (const char *)a.src + (size_t)c0 * es;
    c.src_ld = a.src_ld > 0 ? a.src_ld : full;
    c.dst = (char *)a.dst + (size_t)c0 * (a.epi == IT_EPI_RAW_F32 ? 4 : es);
    c.dst_ld = a.dst_ld > 0 ? a.dst_ld : full;
    c.self_term = a.self_term ? (const char *)a.self_term + (size_t)c0 * es : nullptr;
    c.self_ld = a.self_ld > 0 ? a.self_ld : full;
    c.bias = a.bias ? a.bias + c0 : nullptr;
    IT_TRY(launch_gather_chunk(c, st));
    c0 += c.dim;
  }
  return IT_OK;
}
