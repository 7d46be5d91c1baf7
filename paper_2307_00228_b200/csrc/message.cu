// Elementwise kernels around the gather:
//   * the learned message of every edge, m_j = act(P[u_j] + Q[j]) (the source part P was computed once per vertex, the
//     edge part Q once per edge, both by the dense transform), written over Q so that the per-edge-row gather can
//     reduce it; or, where the product that makes Q finishes and reduces the messages itself (bf16), the two small kernels
//     around it: the first vertex of every tile of edges, and the vertices that cross tiles;
//   * for GAT layers whose logits read the edge features: the message row of every edge (a copy of its source's row)
//     and its logit term per head (source score + the edge's share), so that the reduce can walk rows in edge order;
//   * the receiver's finish of a partial-gather over source partitions (scale, zero the vertices without in-edges,
//     round to the storage type).
// All are HBM-bound streams of 16-byte slices; the only irregular access is the source row of an edge.
#include "common.cuh"

namespace {

constexpr int MSG_THREADS = 256;
constexpr int MSG_UNROLL = 4;   // slices in flight per thread

__device__ __forceinline__ float msg_act(float x, int act) {
  if (act == IT_ACT_RELU) return fmaxf(x, 0.f);
  if (act == IT_ACT_ELU) return it_elu(x);
  return x;
}

// 16 bytes of a row: four fp32 or eight bf16 values
template <typename T>
__device__ __forceinline__ uint4 add_act_slice(const uint4 &p, const uint4 &q, int act) {
  const uint32_t pw[4] = {p.x, p.y, p.z, p.w}, qw[4] = {q.x, q.y, q.z, q.w};
  uint32_t o[4];
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int i = 0; i < 4; ++i) o[i] = __float_as_uint(msg_act(__uint_as_float(pw[i]) + __uint_as_float(qw[i]), act));
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float lo = msg_act(__uint_as_float(pw[i] << 16) + __uint_as_float(qw[i] << 16), act);
      const float hi = msg_act(__uint_as_float(pw[i] & 0xffff0000u) + __uint_as_float(qw[i] & 0xffff0000u), act);
      __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
      o[i] = *reinterpret_cast<uint32_t *>(&h);
    }
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// slices: 16-byte slices per row; total = n_edges * slices
template <typename T>
__global__ void __launch_bounds__(MSG_THREADS) edge_messages_kernel(const int32_t *__restrict__ indices, const uint4 *__restrict__ P,
                                                                    uint4 *__restrict__ M, int64_t total, int slices, int act) {
  const int64_t stride = (int64_t)gridDim.x * MSG_THREADS;
  for (int64_t t0 = (int64_t)blockIdx.x * MSG_THREADS + threadIdx.x; t0 < total; t0 += stride * MSG_UNROLL) {
    uint4 p[MSG_UNROLL], q[MSG_UNROLL];
#pragma unroll
    for (int u = 0; u < MSG_UNROLL; ++u) {
      const int64_t t = t0 + u * stride;
      if (t < total) {
        const int64_t j = t / slices;
        const int c = (int)(t - j * slices);
        const int64_t src = __ldg(indices + j);
        p[u] = __ldg(P + src * slices + c);
        q[u] = __ldcs(M + t);
      }
    }
#pragma unroll
    for (int u = 0; u < MSG_UNROLL; ++u) {
      const int64_t t = t0 + u * stride;
      if (t < total) __stcs(M + t, add_act_slice<T>(p[u], q[u], act));
    }
  }
}

// GAT with edge features: the message row of every edge (a copy of its source's row, so that the reduce can walk rows
// in edge order) ...
__global__ void __launch_bounds__(MSG_THREADS) gat_edge_rows_kernel(const int32_t *__restrict__ indices, const uint4 *__restrict__ Z,
                                                                    uint4 *__restrict__ Zj, int64_t total, int slices) {
  const int64_t stride = (int64_t)gridDim.x * MSG_THREADS;
  for (int64_t t0 = (int64_t)blockIdx.x * MSG_THREADS + threadIdx.x; t0 < total; t0 += stride * MSG_UNROLL) {
    uint4 z[MSG_UNROLL];
#pragma unroll
    for (int u = 0; u < MSG_UNROLL; ++u) {
      const int64_t t = t0 + u * stride;
      if (t < total) {
        const int64_t j = t / slices;
        z[u] = __ldg(Z + (int64_t)__ldg(indices + j) * slices + (t - j * slices));
      }
    }
#pragma unroll
    for (int u = 0; u < MSG_UNROLL; ++u) {
      const int64_t t = t0 + u * stride;
      if (t < total) __stcs(Zj + t, z[u]);
    }
  }
}
// ... and its logit term per head: the source's score plus the edge's own share att_edge[h] . e_j
template <typename T>
__global__ void __launch_bounds__(MSG_THREADS) gat_edge_scores_kernel(const int32_t *__restrict__ indices, const float *__restrict__ scores,
                                                                      const T *__restrict__ ef, const float *__restrict__ att_edge,
                                                                      float *__restrict__ sc, int64_t n_edges, int heads, int edge_dim) {
  const int64_t total = n_edges * heads, stride = (int64_t)gridDim.x * MSG_THREADS;
  for (int64_t t = (int64_t)blockIdx.x * MSG_THREADS + threadIdx.x; t < total; t += stride) {
    const int64_t j = t / heads;
    const int h = (int)(t - j * heads);
    float acc = 0.f;
    for (int k = 0; k < edge_dim; ++k) {
      float e;
      if constexpr (sizeof(T) == 4) e = __ldg(reinterpret_cast<const float *>(ef) + j * edge_dim + k);
      else e = __bfloat162float(ef[j * edge_dim + k]);
      acc = fmaf(__ldg(att_edge + h * edge_dim + k), e, acc);
    }
    sc[t] = __ldg(scores + (int64_t)__ldg(indices + j) * (2 * heads) + h) + acc;
  }
}

// The same for 1, 2, 4 or 8 heads and rows of 16-byte pieces: one thread per edge, its feature row in 16-byte loads, all heads
// at once, the attention vectors in shared memory.  (A thread per edge and head with scalar loads took 390 us for 8M edges of 16
// fp32 features and 4 heads: now 152.)
template <typename T, int H>
__global__ void __launch_bounds__(MSG_THREADS) gat_edge_scores_wide_kernel(const int32_t *__restrict__ indices, const float *__restrict__ scores,
                                                                           const uint4 *__restrict__ ef, const float *__restrict__ att_edge,
                                                                           float *__restrict__ sc, int64_t n_edges, int edge_dim) {
  constexpr int PER = 16 / (int)sizeof(T);   // features of a piece
  extern __shared__ float att[];             // [edge_dim][H]
  for (int i = threadIdx.x; i < edge_dim * H; i += MSG_THREADS) att[i] = att_edge[(i % H) * edge_dim + i / H];
  __syncthreads();
  const int pieces = edge_dim / PER;
  const int64_t stride = (int64_t)gridDim.x * MSG_THREADS;
  for (int64_t j = (int64_t)blockIdx.x * MSG_THREADS + threadIdx.x; j < n_edges; j += stride) {
    const float *src = scores + (int64_t)__ldcs(indices + j) * (2 * H);
    float acc[H];
#pragma unroll
    for (int h = 0; h < H; ++h) acc[h] = 0.f;
    const uint4 *row = ef + j * pieces;
#pragma unroll 4
    for (int q = 0; q < pieces; ++q) {
      const uint4 x = __ldg(row + q);
      const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int i = 0; i < PER; ++i) {
        float e;
        if constexpr (sizeof(T) == 4) e = __uint_as_float(w[i]);
        else e = __uint_as_float((i & 1) ? (w[i / 2] & 0xffff0000u) : (w[i / 2] << 16));
#pragma unroll
        for (int h = 0; h < H; ++h) acc[h] = fmaf(att[(q * PER + i) * H + h], e, acc[h]);
      }
    }
#pragma unroll
    for (int h = 0; h < H; ++h) acc[h] += __ldg(src + h);
    if constexpr (H >= 4) {
#pragma unroll
      for (int h = 0; h < H; h += 4) __stcs(reinterpret_cast<float4 *>(sc + j * H + h), make_float4(acc[h], acc[h + 1], acc[h + 2], acc[h + 3]));
    } else if constexpr (H == 2) {
      __stcs(reinterpret_cast<float2 *>(sc + j * 2), make_float2(acc[0], acc[1]));
    } else {
      __stcs(sc + j, acc[0]);
    }
  }
}

__global__ void __launch_bounds__(MSG_THREADS) compact_scores_kernel(const float *__restrict__ scores, float *__restrict__ dense,
                                                                     int64_t total, int heads) {
  const int64_t stride = (int64_t)gridDim.x * MSG_THREADS;
  for (int64_t t = (int64_t)blockIdx.x * MSG_THREADS + threadIdx.x; t < total; t += stride) {
    const int64_t v = t / heads;
    dense[t] = __ldcs(scores + v * 2 * heads + (t - v * heads));
  }
}

// one thread per four consecutive entries of a row
template <typename T>
__global__ void __launch_bounds__(MSG_THREADS) aggregate_finish_kernel(const float4 *__restrict__ raw, const float *__restrict__ scale,
                                                                       T *__restrict__ out, int64_t total4, int quads) {
  const int64_t stride = (int64_t)gridDim.x * MSG_THREADS;
  for (int64_t t = (int64_t)blockIdx.x * MSG_THREADS + threadIdx.x; t < total4; t += stride) {
    const int64_t v = t / quads;
    const float s = __ldg(scale + v);
    float4 x = __ldcs(raw + t);
    if (s == 0.f) x = make_float4(0.f, 0.f, 0.f, 0.f);
    else { x.x *= s; x.y *= s; x.z *= s; x.w *= s; }
    if constexpr (sizeof(T) == 4) {
      reinterpret_cast<float4 *>(out)[t] = x;
    } else {
      __nv_bfloat162 a = __floats2bfloat162_rn(x.x, x.y), b = __floats2bfloat162_rn(x.z, x.w);
      reinterpret_cast<uint2 *>(out)[t] = make_uint2(*reinterpret_cast<uint32_t *>(&a), *reinterpret_cast<uint32_t *>(&b));
    }
  }
}

// ----------------------------------------------------------------------------- messages reduced by their product
__device__ __forceinline__ int64_t bound_of(const void *indptr, int is64, int64_t v) {
  return is64 ? (int64_t)__ldg(reinterpret_cast<const long long *>(indptr) + v) : (int64_t)__ldg(reinterpret_cast<const int32_t *>(indptr) + v);
}

// tile_first[t]: the vertex that edge IT_MSG_TILE * t belongs to; ends[j]: the vertex whose last edge j is (the others: cleared
// before).  A thread per vertex; vertices of several tiles by the whole warp.  Bound by clearing the ends and reading indptr once.
__global__ void __launch_bounds__(MSG_THREADS) message_tiles_kernel(const void *indptr, int is64, int64_t n, int32_t *__restrict__ tile_first,
                                                                 int32_t *__restrict__ ends) {
  const int lane = threadIdx.x & 31;
  for (int64_t v0 = ((int64_t)blockIdx.x * MSG_THREADS + threadIdx.x) - lane; v0 < n; v0 += (int64_t)gridDim.x * MSG_THREADS) {
    const int64_t v = v0 + lane;
    int64_t t0 = 0, count = 0;
    if (v < n) {
      const int64_t a = bound_of(indptr, is64, v), b = bound_of(indptr, is64, v + 1);
      t0 = (a + IT_MSG_TILE - 1) / IT_MSG_TILE;
      if (b > a) { count = (b - 1) / IT_MSG_TILE - t0 + 1; ends[b - 1] = (int32_t)v; }
    }
    if (count == 1) tile_first[t0] = (int32_t)v;
    for (unsigned many = __ballot_sync(0xffffffffu, count > 1); many; many &= many - 1) {
      const int l = __ffs(many) - 1;
      const int64_t at = __shfl_sync(0xffffffffu, t0, l), c = __shfl_sync(0xffffffffu, count, l);
      for (int64_t k = lane; k < c; k += 32) tile_first[at + k] = (int32_t)(v0 + l);
    }
  }
}

// The vertices that cross tiles, found at the tile after the one where they begin.  A warp looks at 32 tiles at once and folds the
// parts of their vertices, two vertices of two tiles at a time; the whole block folds a vertex of many.  Parts are folded in edge
// order.  Bound by the trips first vertex -> its bounds -> its parts, made once for 32 tiles (one tile per warp: 114 us for 125k).
constexpr int MSG_JOIN_THREADS = 1024, MSG_JOIN_WARPS = MSG_JOIN_THREADS / 32, MSG_JOIN_BLOCK = 48 /* parts from which on a block takes a vertex */;
__global__ void __launch_bounds__(MSG_JOIN_THREADS, 1) message_combine_kernel(it_tc_reduce q, int64_t n_tiles) {
  __shared__ float4 part[MSG_JOIN_WARPS][32];
  __shared__ int64_t todo[MSG_JOIN_THREADS];
  __shared__ int n_todo;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = lane * 4;
  const bool is_max = q.mode == IT_MSG_WMAX || q.mode == IT_MSG_MAX, is_min = q.mode == IT_MSG_WMIN || q.mode == IT_MSG_MIN;
  const float id = is_max ? -INFINITY : (is_min ? INFINITY : 0.f);
  auto fold = [&](float4 &a, const float4 &y) {
    if (is_max) { a.x = fmaxf(a.x, y.x); a.y = fmaxf(a.y, y.y); a.z = fmaxf(a.z, y.z); a.w = fmaxf(a.w, y.w); }
    else if (is_min) { a.x = fminf(a.x, y.x); a.y = fminf(a.y, y.y); a.z = fminf(a.z, y.z); a.w = fminf(a.w, y.w); }
    else { a.x += y.x; a.y += y.y; a.z += y.z; a.w += y.w; }
  };
  // the parts of the vertex that begins in tile b - 1: part 0 lies there, part k in tile b - 1 + k
  auto load = [&](int64_t b, int64_t k) { return __ldcs(reinterpret_cast<const float4 *>(q.partial + ((b - 1 + k) * 2 + (k == 0 ? 1 : 0)) * q.dim + c)); };
  auto walk = [&](int64_t b, int64_t k0, int64_t k1) {
    float4 a = make_float4(id, id, id, id);
    if (c >= q.dim) return a;
    int64_t k = k0;
    for (; k + 8 <= k1; k += 8) {
      float4 y[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) y[u] = load(b, k + u);
#pragma unroll
      for (int u = 0; u < 8; ++u) fold(a, y[u]);
    }
    for (; k < k1; ++k) fold(a, load(b, k));
    return a;
  };
  auto finish = [&](int64_t v, int64_t deg, float4 a) {
    if (c >= q.dim) return;
    if (q.is_mean) { const float inv = 1.f / (float)deg; a.x *= inv; a.y *= inv; a.z *= inv; a.w *= inv; }
    const __nv_bfloat162 h0 = __floats2bfloat162_rn(a.x, a.y), h1 = __floats2bfloat162_rn(a.z, a.w);
    *reinterpret_cast<uint2 *>(reinterpret_cast<__nv_bfloat16 *>(q.dst) + v * q.dst_ld + c) =
        make_uint2(*reinterpret_cast<const uint32_t *>(&h0), *reinterpret_cast<const uint32_t *>(&h1));
  };
  for (int64_t b0 = 1 + (int64_t)blockIdx.x * MSG_JOIN_THREADS; b0 < n_tiles; b0 += (int64_t)gridDim.x * MSG_JOIN_THREADS) {
    if (threadIdx.x == 0) n_todo = 0;
    __syncthreads();
    const int64_t b = b0 + threadIdx.x;
    int64_t v = 0, deg = 0, parts = 0;   // 0 parts: no vertex begins in tile b - 1 and goes on in tile b
    if (b < n_tiles) {
      v = __ldg(q.tile_first + b);
      const int64_t s = bound_of(q.indptr, q.indptr64, v), e = bound_of(q.indptr, q.indptr64, v + 1);
      if (s < b * IT_MSG_TILE && s >= (b - 1) * IT_MSG_TILE) { parts = (e - 1) / IT_MSG_TILE - b + 2; deg = e - s; }
    }
    if (parts >= MSG_JOIN_BLOCK) todo[atomicAdd(&n_todo, 1)] = b;
    const int64_t wb = b - lane;
    for (unsigned two = __ballot_sync(0xffffffffu, parts == 2); two;) {
      float4 x[2], y[2];
      int l[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        l[u] = two ? __ffs(two) - 1 : -1;
        two &= two - 1;   // (0 stays 0)
        if (l[u] >= 0 && c < q.dim) { x[u] = load(wb + l[u], 0); y[u] = load(wb + l[u], 1); }
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int64_t vv = __shfl_sync(0xffffffffu, v, l[u] & 31), dd = __shfl_sync(0xffffffffu, deg, l[u] & 31);
        if (l[u] < 0) continue;
        fold(x[u], y[u]);
        finish(vv, dd, x[u]);
      }
    }
    for (unsigned some = __ballot_sync(0xffffffffu, parts > 2 && parts < MSG_JOIN_BLOCK); some; some &= some - 1) {
      const int l = __ffs(some) - 1;
      const int64_t vv = __shfl_sync(0xffffffffu, v, l), dd = __shfl_sync(0xffffffffu, deg, l), pp = __shfl_sync(0xffffffffu, parts, l);
      finish(vv, dd, walk(wb + l, 0, pp));
    }
    __syncthreads();
    const int n = n_todo;
    for (int i = 0; i < n; ++i) {
      const int64_t tb = todo[i], tv = __ldg(q.tile_first + tb), s = bound_of(q.indptr, q.indptr64, tv), e = bound_of(q.indptr, q.indptr64, tv + 1);
      const int64_t all = (e - 1) / IT_MSG_TILE - tb + 2, per = (all + MSG_JOIN_WARPS - 1) / MSG_JOIN_WARPS;
      const int64_t k0 = warp * per < all ? warp * per : all, k1 = k0 + per < all ? k0 + per : all;
      part[warp][lane] = walk(tb, k0, k1);
      __syncthreads();
      if (warp == 0) {
        float4 a = part[0][lane];
        for (int w = 1; w < MSG_JOIN_WARPS; ++w) fold(a, part[w][lane]);
        finish(tv, e - s, a);
      }
      __syncthreads();
    }
  }
}

}  // namespace

it_status it_launch_message_tiles(const it_graph *g, int32_t *tile_first, int32_t *ends, cudaStream_t st) {
  if (g->e == 0) return IT_OK;
  IT_CUDA_TRY(cudaMemsetAsync(ends, 0xff, (size_t)((g->e + IT_MSG_TILE - 1) / IT_MSG_TILE) * IT_MSG_TILE * sizeof(int32_t), st));
  const int64_t want = (g->n + MSG_THREADS - 1) / MSG_THREADS, cap = (int64_t)g->num_sms * 8;
  IT_LAUNCH(IT_K_EDGE_MSG, (double)g->n * (g->indptr_type == IT_I64 ? 8.0 : 4.0) + (double)g->e / IT_MSG_TILE * 4.0, 0, st,
            message_tiles_kernel<<<(unsigned)(want < cap ? want : cap), MSG_THREADS, 0, st>>>(g->indptr, g->indptr_type == IT_I64, g->n, tile_first, ends));
  IT_CUDA_TRY(cudaGetLastError());
  return IT_OK;
}

it_status it_launch_message_combine(const it_graph *g, const it_tc_reduce &q, cudaStream_t st) {
  const int64_t tiles = (g->e + IT_MSG_TILE - 1) / IT_MSG_TILE;
  if (tiles > 1) {
    const int64_t want = (tiles - 1 + MSG_JOIN_THREADS - 1) / MSG_JOIN_THREADS, cap = (int64_t)g->num_sms;
    IT_LAUNCH(IT_K_COMBINE, (double)tiles * (2.0 * q.dim * 4.0 + q.dim * 2.0), 0, st,
              message_combine_kernel<<<(unsigned)(want < cap ? want : cap), MSG_JOIN_THREADS, 0, st>>>(q, tiles));
    IT_CUDA_TRY(cudaGetLastError());
  }
  if (g->h_list_offsets[1] > g->h_list_offsets[0]) {   // the vertices without edges
    it_empty_rows_args er{};
    er.g = g; er.row_lo = g->h_list_offsets[0]; er.row_hi = g->h_list_offsets[1];
    er.kind = IT_EMPTY_VALUE; er.dst = q.dst; er.dim = q.dim; er.dtype = IT_BF16; er.pitch = (int64_t)q.dst_ld * 2; er.value = 0.f;
    er.act = IT_ACT_NONE;
    IT_TRY(it_launch_empty_rows(er, IT_K_GATHER_EMPTY, (double)(er.row_hi - er.row_lo) * (16.0 + q.dim * 2.0), st));
  }
  return IT_OK;
}

it_status it_launch_edge_messages(const it_graph *g, it_dtype dtype, int dim, const void *P, void *M, it_act act, cudaStream_t st) {
  const int es = it_dtype_size(dtype);
  IT_REQUIRE(dim > 0 && (dim * es) % 16 == 0, IT_ERR_INVALID_ARG, "edge messages: a row of %d bytes is not a multiple of 16", dim * es);
  if (g->e == 0) return IT_OK;
  const int slices = dim * es / 16;
  const int64_t total = g->e * slices;
  const int64_t want = (total + (int64_t)MSG_THREADS * MSG_UNROLL - 1) / ((int64_t)MSG_THREADS * MSG_UNROLL);
  const int64_t cap = (int64_t)g->num_sms * 16;
  const unsigned blocks = (unsigned)(want < cap ? want : cap);
  // per edge: its index, one row of P (read), one row of Q (read) and the message (written)
  const double bytes = (double)g->e * (4.0 + 3.0 * dim * es);
  if (dtype == IT_F32)
    IT_LAUNCH(IT_K_EDGE_MSG, bytes, 0, st, edge_messages_kernel<float><<<blocks, MSG_THREADS, 0, st>>>(
        g->indices, reinterpret_cast<const uint4 *>(P), reinterpret_cast<uint4 *>(M), total, slices, (int)act));
  else
    IT_LAUNCH(IT_K_EDGE_MSG, bytes, 0, st, edge_messages_kernel<__nv_bfloat16><<<blocks, MSG_THREADS, 0, st>>>(
        g->indices, reinterpret_cast<const uint4 *>(P), reinterpret_cast<uint4 *>(M), total, slices, (int)act));
  IT_CUDA_TRY(cudaGetLastError());
  return IT_OK;
}

it_status it_launch_gat_edge_rows(const it_graph *g, it_dtype dtype, int dim, int heads, const void *Z, const float *scores,
                                  const float *att_edge, void *Zj, float *sc, cudaStream_t st) {
  if (g->e == 0) return IT_OK;
  const int es = it_dtype_size(dtype);
  const int slices = dim * es / 16;
  const int64_t total = g->e * slices;
  const int64_t cap = (int64_t)g->num_sms * 16;
  int64_t want = (total + (int64_t)MSG_THREADS * MSG_UNROLL - 1) / ((int64_t)MSG_THREADS * MSG_UNROLL);
  unsigned blocks = (unsigned)(want < cap ? want : cap);
  if (Zj) IT_LAUNCH(IT_K_EDGE_MSG, (double)g->e * (4.0 + 2.0 * dim * es), 0, st,
            gat_edge_rows_kernel<<<blocks, MSG_THREADS, 0, st>>>(g->indices, reinterpret_cast<const uint4 *>(Z), reinterpret_cast<uint4 *>(Zj), total, slices));
  want = (g->e * heads + MSG_THREADS - 1) / MSG_THREADS;
  blocks = (unsigned)(want < cap ? want : cap);
  const size_t att_bytes = (size_t)heads * g->edge_dim * sizeof(float);
  if ((heads == 1 || heads == 2 || heads == 4 || heads == 8) && att_bytes <= 32 * 1024) {
    const int64_t w2 = (g->e + MSG_THREADS - 1) / MSG_THREADS, cap2 = (int64_t)g->num_sms * 8;
    const unsigned blocks2 = (unsigned)(w2 < cap2 ? w2 : cap2);
    auto go = [&]<typename T, int H>() {
      IT_LAUNCH(IT_K_EDGE_MSG, (double)g->e * (4.0 + (double)g->edge_dim * es + 8.0 * heads), 0, st,
                gat_edge_scores_wide_kernel<T, H><<<blocks2, MSG_THREADS, att_bytes, st>>>(g->indices, scores, reinterpret_cast<const uint4 *>(g->edge_feat), att_edge, sc, g->e, g->edge_dim));
    };
    auto by_heads = [&]<typename T>() {
      if (heads == 1) go.template operator()<T, 1>();
      else if (heads == 2) go.template operator()<T, 2>();
      else if (heads == 4) go.template operator()<T, 4>();
      else go.template operator()<T, 8>();
    };
    if (dtype == IT_F32) by_heads.template operator()<float>();
    else by_heads.template operator()<__nv_bfloat16>();
    IT_CUDA_TRY(cudaGetLastError());
    return IT_OK;
  }
  const double sbytes = (double)g->e * (4.0 + (double)g->edge_dim * es + 8.0 * heads);
  if (dtype == IT_F32)
    IT_LAUNCH(IT_K_EDGE_MSG, sbytes, 0, st, gat_edge_scores_kernel<float><<<blocks, MSG_THREADS, 0, st>>>(
        g->indices, scores, reinterpret_cast<const float *>(g->edge_feat), att_edge, sc, g->e, heads, g->edge_dim));
  else
    IT_LAUNCH(IT_K_EDGE_MSG, sbytes, 0, st, gat_edge_scores_kernel<__nv_bfloat16><<<blocks, MSG_THREADS, 0, st>>>(
        g->indices, scores, reinterpret_cast<const __nv_bfloat16 *>(g->edge_feat), att_edge, sc, g->e, heads, g->edge_dim));
  IT_CUDA_TRY(cudaGetLastError());
  return IT_OK;
}

it_status it_launch_compact_scores(int64_t n, int heads, const float *scores, float *dense, cudaStream_t st) {
  if (n == 0) return IT_OK;
  const int64_t total = n * heads;
  const int64_t want = (total + MSG_THREADS - 1) / MSG_THREADS, cap = (int64_t)IT_NUM_SMS_FALLBACK * 32;
  IT_LAUNCH(IT_K_EDGE_MSG, (double)n * heads * 12.0, 0, st,
            compact_scores_kernel<<<(unsigned)(want < cap ? want : cap), MSG_THREADS, 0, st>>>(scores, dense, total, heads));
  IT_CUDA_TRY(cudaGetLastError());
  return IT_OK;
}

it_status it_launch_aggregate_finish(int64_t n, int dim, it_dtype dtype, const float *raw, const float *scale, void *out, cudaStream_t st) {
  IT_REQUIRE(dim > 0 && dim % 4 == 0, IT_ERR_INVALID_ARG, "aggregate finish: dim %d is not a multiple of 4", dim);
  if (n == 0) return IT_OK;
  const int quads = dim / 4;
  const int64_t total4 = n * quads;
  const int64_t want = (total4 + MSG_THREADS - 1) / MSG_THREADS;
  const int64_t cap = (int64_t)IT_NUM_SMS_FALLBACK * 32;
  const unsigned blocks = (unsigned)(want < cap ? want : cap);
  const double bytes = (double)n * (4.0 + dim * (4.0 + it_dtype_size(dtype)));
  if (dtype == IT_F32)
    IT_LAUNCH(IT_K_AGG_FINISH, bytes, 0, st, aggregate_finish_kernel<float><<<blocks, MSG_THREADS, 0, st>>>(
        reinterpret_cast<const float4 *>(raw), scale, reinterpret_cast<float *>(out), total4, quads));
  else
    IT_LAUNCH(IT_K_AGG_FINISH, bytes, 0, st, aggregate_finish_kernel<__nv_bfloat16><<<blocks, MSG_THREADS, 0, st>>>(
        reinterpret_cast<const float4 *>(raw), scale, reinterpret_cast<__nv_bfloat16 *>(out), total4, quads));
  IT_CUDA_TRY(cudaGetLastError());
  return IT_OK;
}
