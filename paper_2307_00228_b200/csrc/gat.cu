// GAT reduce: per destination and head, e = LeakyReLU(s_src[u] + s_dst[v]), softmax over the
// in-edges, attention-weighted sum of the source rows z_u, then bias and activation.
// One pass over the edges with a running (max, sum, weighted accumulator) state per lane
// ("online" softmax).  Such states merge associatively — (m, l, acc) and (m', l', acc') give
// M = max(m, m'), l e^(m-M) + l' e^(m'-M), acc e^(m-M) + acc' e^(m'-M) — so the groups of a split
// hub are reduced independently into partial states and merged in edge order, exactly like
// the partial sums of the plain gather.  The edge streaming lives in stream.cuh.
#include <type_traits>

#include "stream.cuh"

namespace {

using namespace it_stream;

__host__ __device__ inline int gat_partial_stride(int dim, int heads) { return dim + ((2 * heads + 3) / 4) * 4; }

template <typename T, int SB>
struct GatPolicy {
  using Slice = RowSlice<T, SB>;
  static constexpr int VEC = Slice::VEC;
  static constexpr int NS = VEC + 2;   // accumulators, running max, running sum
  static constexpr bool WEIGHTED = false, HAS_EXTRA = true, NEEDS_OWNER = true, NULLABLE = false;
  const float *__restrict__ scores;    // [n_src, 2*heads]: source scores of the vertex, then its destination scores
  const float *__restrict__ scores_dst;   // the same rows, counted from the first local destination
  const float *__restrict__ bias;
  void *__restrict__ dst;
  float *__restrict__ partials;        // [n_partial_rows, stride]: acc[dim], m[heads], l[heads]
  int dim, heads, head_dim, act;
  int src_stride;                      // floats from one row of `scores` to the next (2*heads; heads when the rows are per edge)
  float slope;
  // per-thread
  int col, head;
  float s_dst;
  uint32_t bias_s;   // shared-window address of a copy of the bias (0: none; read it from global memory)

  void empty_rows(it_empty_rows_args &a) const {
    a.kind = IT_EMPTY_BIAS;
    a.dst = dst; a.dim = dim; a.dtype = sizeof(T) == 4 ? IT_F32 : IT_BF16; a.pitch = (int64_t)dim * (int)sizeof(T);
    a.self = nullptr; a.self_pitch = 0; a.value = 0.f; a.bias = bias; a.act = (it_act)act;
  }
  __device__ __forceinline__ void setup(int t) { col = t * VEC; head = col / head_dim; s_dst = 0.f; }
  __device__ __forceinline__ void init(float (&st)[NS]) const {
#pragma unroll
    for (int k = 0; k < VEC; ++k) st[k] = 0.f;
    st[VEC] = -INFINITY;
    st[VEC + 1] = 0.f;
  }
  __device__ __forceinline__ float extra(uint32_t s) const { return __ldg(scores + (uint64_t)s * src_stride + head); }
  __device__ __forceinline__ const float *extra_ptr(uint32_t s) const { return scores + (uint64_t)s * src_stride + head; }
  __device__ __forceinline__ void edge(float (&st)[NS], const typename Slice::Raw &raw, float, float x) const {
    float e = x + s_dst;
    e = e > 0.f ? e : slope * e;
    // One exponential per edge: of the two factors exp(m - m_new) and exp(e - m_new) one is exp(0) = 1 and the other is
    // exp(-|e - m|).  (First edge: m = -inf, the old state is scaled by exp(-inf) = 0.)
    const float d = e - st[VEC];
    const float t = __expf(-fabsf(d));
    const bool up = d > 0.f;
    const float scale = up ? t : 1.f, pw = up ? 1.f : t;
    const float m_new = up ? e : st[VEC];
    float f[VEC];
    Slice::unpack(raw, f);
    if constexpr (VEC % 2 == 0) {
#pragma unroll
      for (int k = 0; k < VEC; k += 2) scale_fma_f32x2(st[k], st[k + 1], scale, pw, f[k], f[k + 1]);
    } else {
#pragma unroll
      for (int k = 0; k < VEC; ++k) st[k] = fmaf(pw, f[k], st[k] * scale);
    }
    st[VEC + 1] = fmaf(st[VEC + 1], scale, pw);
    st[VEC] = m_new;
  }
  __device__ __forceinline__ void merge(float (&st)[NS], const float (&o)[NS]) const {
    const float m_new = fmaxf(st[VEC], o[VEC]);
    const float f1 = st[VEC] == -INFINITY ? 0.f : __expf(st[VEC] - m_new);
    const float f2 = o[VEC] == -INFINITY ? 0.f : __expf(o[VEC] - m_new);
#pragma unroll
    for (int k = 0; k < VEC; ++k) st[k] = st[k] * f1 + o[k] * f2;
    st[VEC + 1] = st[VEC + 1] * f1 + o[VEC + 1] * f2;
    st[VEC] = m_new;
  }
  __device__ __forceinline__ void begin_row(int32_t, int32_t owner) {
    s_dst = __ldg(scores_dst + (int64_t)owner * (2 * heads) + heads + head);
  }
  __device__ __forceinline__ void end_row(float (&st)[NS], int32_t dest, int32_t, int64_t) const {
    if (dest < 0) {   // a group of a split vertex: its state goes to the partial buffer
      float *q = partials + (int64_t)(~dest) * gat_partial_stride(dim, heads);
      float a[VEC];
#pragma unroll
      for (int i = 0; i < VEC; ++i) a[i] = st[i];
      store_floats<VEC>(q + col, a);
      if (col % head_dim == 0) {
        q[dim + head] = st[VEC];
        q[dim + heads + head] = st[VEC + 1];
      }
      return;
    }
    const float inv = st[VEC + 1] > 0.f ? 1.f / st[VEC + 1] : 0.f;
    float o[VEC];
#pragma unroll
    for (int i = 0; i < VEC; ++i) o[i] = 0.f;
    if (bias_s != 0) {
#pragma unroll
      for (int i = 0; i < VEC; i += 4) {   // (only set for 16-byte slices: four columns at a time)
        const uint4 b = lds_slice<16>(bias_s + (uint32_t)(col + i) * 4);
        o[i] = __uint_as_float(b.x);
        if (i + 3 < VEC) { o[i + 1] = __uint_as_float(b.y); o[i + 2] = __uint_as_float(b.z); o[i + 3] = __uint_as_float(b.w); }
      }
    } else if (bias) {
#pragma unroll
      for (int i = 0; i < VEC; ++i) o[i] = __ldg(bias + col + i);
    }
#pragma unroll
    for (int i = 0; i < VEC; ++i) o[i] = fmaf(st[i], inv, o[i]);
    act_slice<VEC>(o, act);
    Slice::store(reinterpret_cast<T *>(dst) + (int64_t)dest * dim + col, o);
  }
};

}  // namespace

#include "gat_rows.cuh"

namespace {

// Merge the partial states of every long vertex in edge order: one block per vertex, lane = C consecutive columns of one head
// (four where a head's width allows it: one pass over the partial rows of up to 128 columns); every warp merges a contiguous
// range of the pieces, four in flight, the warps' states follow in warp order.  (One column per lane and two passes over each
// took 465 us for the two layers of 5M vertices / 100M edges: now 176.)
// EDGES: where there is no partial buffer (a layer that just fits the built-in scratch) the same over the vertex's edges, each a state
// of its own: its logit, a weight of 1, its source row.
struct GatCombineParams {
  const int32_t *__restrict__ long_owners;
  const int64_t *__restrict__ piece_ptr;
  const float *__restrict__ partials;
  const float *__restrict__ bias;
  void *__restrict__ dst;
  int64_t n_long;
  int dim, heads, head_dim, act;
  const int64_t *__restrict__ owner_indptr;    // EDGES: the vertex's edges, ...
  const int64_t *__restrict__ shadow_indptr;
  const int32_t *__restrict__ indices;         // ... their sources (NULL: z has a row per edge), ...
  const void *__restrict__ z;                  // ... source rows, ...
  const float *__restrict__ scores;            // ... and logit terms, rows of `stride` by source or by edge; destination scores
  const float *__restrict__ scores_dst;
  int stride, per_edge_scores;
  float slope;
};

// a state of C columns: maximum, sum of weights, weighted sums
template <int C>
struct MergeState {
  float m, l, acc[C];
  __device__ __forceinline__ void clear() {
    m = -INFINITY; l = 0.f;
#pragma unroll
    for (int i = 0; i < C; ++i) acc[i] = 0.f;
  }
  __device__ __forceinline__ void merge(const MergeState &o) {   // o follows in edge order
    const float mm = fmaxf(m, o.m);
    const float f1 = m == -INFINITY ? 0.f : it_exp(m - mm), f2 = o.m == -INFINITY ? 0.f : it_exp(o.m - mm);
    m = mm; l = l * f1 + o.l * f2;
#pragma unroll
    for (int i = 0; i < C; ++i) acc[i] = acc[i] * f1 + o.acc[i] * f2;
  }
};

template <typename T, int C, bool EDGES>
__global__ void __launch_bounds__(THREADS) gat_combine_kernel(GatCombineParams p) {
  using Index = std::conditional_t<EDGES, int64_t, int>;   // (pieces are counted with 31 bits)
  constexpr int WARPS = THREADS / 32;
  __shared__ MergeState<C> red[WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int stride = gat_partial_stride(p.dim, p.heads);
  for (int64_t k = blockIdx.x; k < p.n_long; k += gridDim.x) {
    const int64_t v = __ldg(p.long_owners + k);
    const int64_t p0 = EDGES ? __ldg(p.shadow_indptr + __ldg(p.owner_indptr + v)) : __ldg(p.piece_ptr + k);
    const Index n = (Index)((EDGES ? __ldg(p.shadow_indptr + __ldg(p.owner_indptr + v + 1)) : __ldg(p.piece_ptr + k + 1)) - p0);
    const Index per = (n + WARPS - 1) / WARPS, a = warp * per < n ? warp * per : n, b = a + per < n ? a + per : n;
    for (int c0 = 0; c0 < p.dim; c0 += 32 * C) {
      const int c = c0 + lane * C;
      MergeState<C> s;
      s.clear();
      if (c < p.dim) {
        const int head = c / p.head_dim;
        const float *P = p.partials + p0 * stride;
        const float sd = EDGES ? __ldg(p.scores_dst + v * (2 * p.heads) + p.heads + head) : 0.f;
        auto load = [&](Index g, MergeState<C> &x) {
          if constexpr (EDGES) {
            using Slice = RowSlice<T, C * (int)sizeof(T)>;
            const int64_t j = p0 + (int64_t)g, u = p.indices ? (int64_t)__ldg(p.indices + j) : j;
            const float e = __ldg(p.scores + (p.per_edge_scores ? j : u) * p.stride + head) + sd;
            x.m = e > 0.f ? e : p.slope * e;
            x.l = 1.f;
            Slice::unpack(Slice::load(reinterpret_cast<const char *>(p.z) + (u * p.dim + c) * (int64_t)sizeof(T)), x.acc);
            return;
          }
          const float *row = P + (int64_t)g * stride;
          x.m = __ldg(row + p.dim + head);
          x.l = __ldg(row + p.dim + p.heads + head);
          if constexpr (C == 4) {
            const float4 y = __ldcs(reinterpret_cast<const float4 *>(row + c));
            x.acc[0] = y.x; x.acc[1] = y.y; x.acc[2] = y.z; x.acc[3] = y.w;
          } else {
#pragma unroll
            for (int i = 0; i < C; ++i) x.acc[i] = __ldcs(row + c + i);
          }
        };
        Index g = a;
        auto merge_to = [&](MergeState<C> &t, Index end) {
          for (; g + 4 <= end; g += 4) {
            MergeState<C> x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) load(g + u, x[u]);
#pragma unroll
            for (int u = 0; u < 4; ++u) t.merge(x[u]);
          }
          for (; g < end; ++g) {
            MergeState<C> x;
            load(g, x);
            t.merge(x);
          }
        };
        if constexpr (EDGES) {
          while (g < b) {   // in runs as long as a piece, so that sums are rounded no more often than with partial rows
            MergeState<C> run;
            run.clear();
            merge_to(run, b - g < 512 ? b : g + 512);
            s.merge(run);
          }
        } else {
          merge_to(s, b);
        }
      }
      __syncthreads();   // red free again
      red[warp][lane] = s;
      __syncthreads();
      if (warp != 0 || c >= p.dim) continue;
      for (int w = 1; w < WARPS; ++w) s.merge(red[w][lane]);
      const float inv = s.l > 0.f ? 1.f / s.l : 0.f;
      float o[C];
#pragma unroll
      for (int i = 0; i < C; ++i) o[i] = act_apply(s.acc[i] * inv + (p.bias ? __ldg(p.bias + c + i) : 0.f), p.act);
      RowSlice<T, C * (int)sizeof(T)>::store(reinterpret_cast<T *>(p.dst) + v * p.dim + c, o);
    }
  }
}

template <typename T, int SB>
GatPolicy<T, SB> make_policy(const it_gat_args &a) {
  GatPolicy<T, SB> pol;
  pol.scores = a.src_scores ? a.src_scores : a.scores; pol.src_stride = a.src_scores ? a.heads : 2 * a.heads;
  pol.scores_dst = a.scores_dst ? a.scores_dst : a.scores; pol.bias = a.bias; pol.dst = a.dst; pol.partials = a.partials;
  pol.dim = a.heads * a.head_dim; pol.heads = a.heads; pol.head_dim = a.head_dim; pol.act = a.act; pol.slope = a.slope;
  pol.col = 0; pol.head = 0; pol.s_dst = 0.f; pol.bias_s = 0;
  return pol;
}

// algorithmic bytes: per edge the index, one source score per head and one source row; per row its metadata, owner,
// destination scores and one output row
auto gat_bytes(const it_gat_args &a) {
  const it_graph *g = a.g;
  const int heads = a.heads;
  const double row_bytes = (double)heads * a.head_dim * it_dtype_size(a.dtype);
  return [=](int b, int64_t rows) {
    return (double)g->h_list_edges[b] * (4.0 + 4.0 * heads + row_bytes) + (double)rows * (20.0 + 4.0 * heads + row_bytes);
  };
}

template <typename T, int SB, int LPR>
it_status launch_gat_lpr(const it_gat_args &a, StreamParams sp, cudaStream_t st) {
  return launch_buckets<T, SB, LPR, false>(a.g, sp, make_policy<T, SB>(a), gat_bytes(a), IT_K_GAT_FLAT, IT_K_GAT_EMPTY, a.counters, st);
}

// f.template operator()<LPR, H>() for the shapes that the batched kernels take
template <class F>
it_status dispatch_batched(int row_bytes, int heads, F f) {
  auto by_heads = [&]<int LPR>() -> it_status {
    switch (heads) {
      case 1: return f.template operator()<LPR, 1>();
      case 2: return f.template operator()<LPR, 2>();
      case 4: return f.template operator()<LPR, 4>();
    }
    if constexpr (LPR >= 8) return f.template operator()<LPR, 8>();
    it_set_error("gat: %d heads in a row of %d bytes", heads, row_bytes);   // (not with it_gat_batched())
    return IT_ERR_UNSUPPORTED;
  };
  switch (row_bytes) {
    case 512: return by_heads.template operator()<32>();
    case 256: return by_heads.template operator()<16>();
    case 128: return by_heads.template operator()<8>();
    default: return by_heads.template operator()<4>();
  }
}

template <typename T>
it_status launch_gat(const it_gat_args &a, StreamParams sp, cudaStream_t st) {
  const it_graph *g = a.g;
  const bool whole = !a.partials && g->n_long > 0;   // long vertices are left to the combine
  // A lane of a 128-byte row holds half a head of four or one of eight: a step then computes as many exponentials per lane as the
  // per-edge softmax, and that one has no step to set up.  It wins but for rows of a few edges and, for four heads in bf16, where
  // vertices are gathered in pieces (batched against per edge: bf16 4 heads, 1M vertices of 31 / 40 / 100 edges 1019 / 1343 / 2604
  // against 925 / 1209 / 2410 us, 6M of 2 / 12 / 40 edges 1259 / 3787 / 11039 against 1350 / 3726 / 10030, 1M / 15M power law 549
  // against 566; the same graph, 8 heads, 1266 against 1204, fp32 4 heads 811 against 795, 8 heads 909 against 827).
  const bool per_edge = a.heads * a.head_dim * (int)sizeof(T) == 128 && !a.per_edge_scores && !it_small_graph(g) && g->e > 8 * g->n &&
                        (a.heads == 8 || (a.heads == 4 && (g->n_long == 0 || sizeof(T) == 4)));
  if (!a.per_edge_rows && a.counters && !per_edge && it_gat_batched(a.dtype, a.heads, a.head_dim))
    return dispatch_batched(a.heads * a.head_dim * (int)sizeof(T), a.heads, [&]<int LPR, int H>() {
      if (it_small_graph(a.g) && !whole) return launch_gat_small<T, LPR, H>(a, sp, make_policy<T, 16>(a), st);
      return launch_gat_rows<T, LPR, H>(a, sp, make_policy<T, 16>(a), gat_bytes(a), st);
    });
  // 16-byte slices as long as one never straddles two heads
  const bool wide = (a.head_dim * (int)sizeof(T)) % 16 == 0;
  const int row_bytes = a.heads * a.head_dim * (int)sizeof(T);
  if ((row_bytes & (row_bytes - 1)) != 0 || row_bytes < 16 || row_bytes > 512) {
    it_set_error("feature row of %d bytes is not 16, 32, 64, 128, 256 or 512 bytes", row_bytes);
    return IT_ERR_UNSUPPORTED;
  }
  return dispatch_row_bytes(row_bytes, wide && row_bytes >= 128, [&]<int SB, int LPR>() {
    if ((a.head_dim * (int)sizeof(T)) % SB != 0) {
      it_set_error("gat: a %d-byte lane slice would straddle two heads (head_dim %d)", SB, a.head_dim);
      return IT_ERR_UNSUPPORTED;
    }
    return launch_gat_lpr<T, SB, LPR>(a, sp, st);
  });
}

}  // namespace

bool it_gat_batched(it_dtype dtype, int heads, int head_dim) {
  const int es = it_dtype_size(dtype), row = heads * head_dim * es;
  return (heads == 1 || heads == 2 || heads == 4 || heads == 8) && (head_dim * es) % 16 == 0 && (row == 128 || row == 256 || row == 512 || (row == 64 && heads <= 4));
}

size_t it_gat_partial_bytes(const it_graph *g, int dim, int heads) {
  return (size_t)g->n_partial_rows * gat_partial_stride(dim, heads) * sizeof(float);
}

it_status it_launch_gat(const it_gat_args &a, cudaStream_t st) {
  const it_graph *g = a.g;
  if (g->n == 0) return IT_OK;
  StreamParams sp;
  sp.meta = g->list_meta; sp.owner = g->list_owner; sp.indices = a.per_edge_rows ? nullptr : g->indices; sp.weights = nullptr;
  sp.src = a.z; sp.row_lo = sp.row_hi = 0; sp.dim = a.heads * a.head_dim; sp.batch_rows = 1; sp.counter = nullptr; sp.claim = 1; sp.slices = 0;
  sp.src_pitch = (uint32_t)(sp.dim * it_dtype_size(a.dtype));
  if (a.dtype == IT_F32) IT_TRY(launch_gat<float>(a, sp, st));
  else IT_TRY(launch_gat<__nv_bfloat16>(a, sp, st));
  if (g->n_long > 0 && !(it_small_graph(g) && a.partials && it_gat_batched(a.dtype, a.heads, a.head_dim) && !a.per_edge_rows)) {
    GatCombineParams c;
    c.long_owners = g->long_owners; c.piece_ptr = g->piece_ptr; c.partials = a.partials; c.bias = a.bias;
    c.dst = a.dst; c.n_long = g->n_long; c.dim = a.heads * a.head_dim; c.heads = a.heads;
    c.head_dim = a.head_dim; c.act = a.act;
    const int64_t cap = (int64_t)g->num_sms * 8;
    const unsigned blocks = (unsigned)(g->n_long < cap ? g->n_long : cap);
    c.owner_indptr = g->owner_indptr; c.shadow_indptr = g->shadow_indptr; c.indices = sp.indices; c.z = a.z;
    c.scores = a.src_scores ? a.src_scores : a.scores; c.stride = a.src_scores ? a.heads : 2 * a.heads; c.per_edge_scores = a.per_edge_scores;
    c.scores_dst = a.scores_dst ? a.scores_dst : a.scores; c.slope = a.slope;
    const double es = it_dtype_size(a.dtype);
    const double cbytes = (a.partials ? (double)it_gat_partial_bytes(g, c.dim, c.heads)
                                      : (double)g->h_list_edges[g->n_lists - 1] * (4.0 + 4.0 * c.heads + c.dim * es)) + (double)g->n_long * c.dim * es;
    auto go = [&]<typename T, int C>() {
      if (a.partials) IT_LAUNCH(IT_K_COMBINE, cbytes, 0, st, gat_combine_kernel<T, C, false><<<blocks, THREADS, 0, st>>>(c));
      else IT_LAUNCH(IT_K_COMBINE, cbytes, 0, st, gat_combine_kernel<T, C, true><<<blocks, THREADS, 0, st>>>(c));
    };
    const bool four = a.head_dim % 4 == 0;
    if (a.dtype == IT_F32) { if (four) go.template operator()<float, 4>(); else go.template operator()<float, 1>(); }
    else { if (four) go.template operator()<__nv_bfloat16, 4>(); else go.template operator()<__nv_bfloat16, 2>(); }
    IT_CUDA_TRY(cudaGetLastError());
  }
  return IT_OK;
}
