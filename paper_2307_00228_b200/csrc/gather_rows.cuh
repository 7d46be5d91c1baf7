// Gather: the aggregate over the in-edges of one shadow row (sum / mean / max / min of w_e * h_src).  The edge streaming
// itself lives in stream.cuh; this file supplies the per-lane state and what happens at the end of a row.  Included by
// one source file per storage type (the kernels are many; they compile side by side).
#pragma once
#include "gather_small.cuh"

namespace {

using namespace it_stream;

// Per lane: VEC fp32 accumulators for its slice of the row.

template <typename T, int SB, int RED, bool WEIGHTED_>
struct SagePolicy {
  using Slice = RowSlice<T, SB>;
  static constexpr int VEC = Slice::VEC;
  // Plain max / min of bf16 rows stays packed, two entries per word: a quarter of the instructions (the largest of bf16 values
  // is one of them, so nothing is rounded): extreme hubs, 20M vertices / 200M edges, three layers, 17.4 -> 15.2 ms.
  static constexpr bool PACKED = RED != RED_SUM && !WEIGHTED_ && sizeof(T) == 2 && SB == 16;
  static constexpr int NS = PACKED ? VEC / 2 : VEC;
  static constexpr bool WEIGHTED = WEIGHTED_, HAS_EXTRA = false, NEEDS_OWNER = false, NULLABLE = false;
  float *__restrict__ partials;
  void *__restrict__ dst;
  const void *__restrict__ self_term;
  const float *__restrict__ bias;
  int dim, dst_ld, self_ld, is_mean, epi, act;   // dim: width of this column chunk; *_ld: row lengths of dst / the self term
  // per-thread
  int col;
  float self[VEC];

  __host__ __device__ void empty_rows(it_empty_rows_args &a) const {
    const bool raw = epi == IT_EPI_RAW_F32;
    a.kind = epi == IT_EPI_ADD_ACT ? IT_EMPTY_SELF : (epi == IT_EPI_BIAS_ACT ? IT_EMPTY_BIAS : IT_EMPTY_VALUE);
    a.dst = dst; a.dim = dim; a.dtype = raw || sizeof(T) == 4 ? IT_F32 : IT_BF16; a.pitch = (int64_t)dst_ld * (raw ? 4 : (int)sizeof(T));
    a.self = self_term; a.self_pitch = (int64_t)self_ld * (int)sizeof(T);
    a.value = raw ? (RED == RED_MAX ? -INFINITY : (RED == RED_MIN ? INFINITY : 0.f)) : 0.f;
    a.bias = bias; a.act = (it_act)act;
  }
  __device__ __forceinline__ void setup(int t) { col = t * VEC; }
  static __device__ __forceinline__ float pick2(float a, float b) {   // two bf16 entries per word
    uint32_t r;
    if (RED == RED_MAX) asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(__float_as_uint(a)), "r"(__float_as_uint(b)));
    else asm("min.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(__float_as_uint(a)), "r"(__float_as_uint(b)));
    return __uint_as_float(r);
  }
  __device__ __forceinline__ void init(float (&st)[NS]) const {
    if constexpr (PACKED) {
#pragma unroll
      for (int k = 0; k < NS; ++k) st[k] = __uint_as_float(RED == RED_MAX ? 0xff80ff80u : 0x7f807f80u);   // -inf / +inf
      return;
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) st[k] = RED == RED_MAX ? -INFINITY : (RED == RED_MIN ? INFINITY : 0.f);
  }
  __device__ __forceinline__ float extra(uint32_t) const { return 0.f; }
  __device__ __forceinline__ const float *extra_ptr(uint32_t) const { return nullptr; }
  __device__ __forceinline__ void edge(float (&st)[NS], const typename Slice::Raw &raw, float w, float) const {
    if constexpr (RED == RED_SUM && !WEIGHTED && sizeof(T) == 2 && IT_MIXED_ADD != 0) {
      // bf16 rows, plain sum: the mixed-precision add takes the bf16 operand as it is (same result as widening it first)
      uint32_t w[SB / 4];
      raw_words<SB>(raw, w);
#pragma unroll
      for (int i = 0; i < SB / 4; ++i) add_bf16x2_to_f32(st[2 * i], st[2 * i + 1], w[i]);
      return;
    }
    if constexpr (PACKED) {
      uint32_t q[SB / 4];
      raw_words<SB>(raw, q);
#pragma unroll
      for (int k = 0; k < NS; ++k) st[k] = pick2(st[k], __uint_as_float(q[k]));
      return;
    }
    float f[VEC];
    Slice::unpack(raw, f);
    if constexpr (RED == RED_SUM && !WEIGHTED && VEC % 2 == 0) {   // two accumulators per instruction (measured: 1 % on the
#pragma unroll                                                      // 128-byte rows; with a weight the pair set-up eats the gain)
      for (int k = 0; k < VEC; k += 2) add_f32x2(st[k], st[k + 1], f[k], f[k + 1]);
    } else {
#pragma unroll
      for (int k = 0; k < VEC; ++k) {
        if (RED == RED_MAX) st[k] = fmaxf(st[k], WEIGHTED ? w * f[k] : f[k]);
        else if (RED == RED_MIN) st[k] = fminf(st[k], WEIGHTED ? w * f[k] : f[k]);
        else st[k] = WEIGHTED ? fmaf(w, f[k], st[k]) : st[k] + f[k];
      }
    }
  }
  __device__ __forceinline__ void merge(float (&st)[NS], const float (&o)[NS]) const {
    if constexpr (PACKED) {
#pragma unroll
      for (int k = 0; k < NS; ++k) st[k] = pick2(st[k], o[k]);
      return;
    }
#pragma unroll
    for (int k = 0; k < NS; ++k) st[k] = RED == RED_MAX ? fmaxf(st[k], o[k]) : (RED == RED_MIN ? fminf(st[k], o[k]) : st[k] + o[k]);
  }
  // the matching slice of the self term is fetched when the row starts, so that end_row does not wait for it
  __device__ __forceinline__ void begin_row(int32_t dest, int32_t) {
    if (epi == IT_EPI_ADD_ACT && dest >= 0)
      Slice::unpack(Slice::load_stream(reinterpret_cast<const char *>(self_term) + ((int64_t)dest * self_ld + col) * (int64_t)sizeof(T)), self);
  }
  __device__ __forceinline__ void end_row(float (&packed)[NS], int32_t dest, int32_t, int64_t len) const {
    float st[VEC];
#pragma unroll
    for (int i = 0; i < VEC; ++i) {
      if constexpr (PACKED) st[i] = __uint_as_float((i & 1) ? (__float_as_uint(packed[i / 2]) & 0xffff0000u) : (__float_as_uint(packed[i / 2]) << 16));
      else st[i] = packed[i];
    }
    if (RED != RED_SUM && len == 0 && epi != IT_EPI_RAW_F32) {
#pragma unroll
      for (int i = 0; i < VEC; ++i) st[i] = 0.f;
    }
    if (dest < 0) {  // a group of a split vertex: raw partial, finished by the combine kernel
      store_floats<VEC>(partials + (int64_t)(~dest) * dim + col, st);
      return;
    }
    if (epi == IT_EPI_RAW_F32) {   // one part's share of a partial-gather: the reduce as it is (its identity for an empty row)
      store_floats<VEC>(reinterpret_cast<float *>(dst) + (int64_t)dest * dst_ld + col, st);
      return;
    }
    if (is_mean && len > 0) {
      const float inv = 1.f / (float)len;
#pragma unroll
      for (int i = 0; i < VEC; ++i) st[i] *= inv;
    }
    if (epi == IT_EPI_ADD_ACT) {
#pragma unroll
      for (int i = 0; i < VEC; ++i) st[i] += self[i];
      act_slice<VEC>(st, act);
    } else if (epi == IT_EPI_BIAS_ACT) {
#pragma unroll
      for (int i = 0; i < VEC; ++i) st[i] += bias ? __ldg(bias + col + i) : 0.f;
      act_slice<VEC>(st, act);
    }
    Slice::store(reinterpret_cast<T *>(dst) + (int64_t)dest * dst_ld + col, st);
  }
};

template <typename T, int SB, int RED, bool WEIGHTED>
SagePolicy<T, SB, RED, WEIGHTED> make_policy(const it_gather_args &a) {
  SagePolicy<T, SB, RED, WEIGHTED> pol;
  pol.partials = a.partials; pol.dst = a.dst; pol.self_term = a.self_term; pol.bias = a.bias; pol.dim = a.dim; pol.dst_ld = a.dst_ld > 0 ? a.dst_ld : a.dim; pol.self_ld = a.self_ld > 0 ? a.self_ld : a.dim;
  pol.is_mean = a.op == IT_GATHER_MEAN && a.epi != IT_EPI_RAW_F32; pol.epi = a.epi; pol.act = a.act; pol.col = 0;
  return pol;
}

// ----------------------------------------------------------------------------- small graphs: every list of a layer in one kernel
// The weighted policy for graphs with and without weights (a weight of 1 changes no result).
template <typename T, int RED>
struct SmallPolicy : SagePolicy<T, 16, RED, true> {
  static constexpr bool NULLABLE = true;
};

template <typename T, int LPR, class Policy>
__global__ void __launch_bounds__(THREADS, SMALL_BLOCKS) gather_small_kernel(StreamParams p, Policy pol, PieceParams q, SmallShare sh, const int64_t *__restrict__ owner_indptr,
                                                                          const int64_t *__restrict__ shadow_indptr) {
  constexpr int SL = 32 / LPR, U = LPR < 4 ? LPR : 4;   // edge slots; rows in flight per lane (SL * U <= 32; eight spill)
  constexpr int LPRS = LPR < 8 ? 8 : LPR;               // lane group of a short row
  constexpr int NS = Policy::NS;
  using Slice = typename Policy::Slice;
  extern __shared__ uint4 small_stage[];
  it_allow_next();
  const int lane = threadIdx.x & 31, slot = lane / LPR, t = lane % LPR;
  const bool active = t < p.slices;
  pol.setup(t);
  const char *my_src = reinterpret_cast<const char *>(p.src) + (size_t)t * 16;
  it_wait_prior();
  if ((int)blockIdx.x < sh.short_blocks) {
    p.row_lo = sh.short_lo; p.row_hi = sh.short_hi;
    if constexpr (LPR <= 16) short_rows_pipe<T, LPRS, Policy, true>(p, pol, blockIdx.x, sh.short_blocks, small_stage);
    return;
  }
  if ((int)blockIdx.x < sh.short_blocks + sh.empty_blocks) {
    it_empty_rows_args a;
    pol.empty_rows(a);
    const EmptyRowsParams er{p.meta, 0, sh.short_lo, (char *)a.dst, (const char *)a.self, a.pitch, a.self_pitch, (int)a.kind,
                             a.dim * (a.dtype == IT_F32 ? 4 : 2) / 16, a.dtype == IT_BF16, (int)a.act, a.value, a.bias};
    small_empties(sh, [&](int b, int n) { empty_rows_warp(er, b, n, lane, [&](int s) { return empty_piece(er, s); }); });
    return;
  }
  small_walk<true, false>(p, sh, lane, [&](const SmallRow &m, int32_t idx, float w) {
    float st[NS];
    pol.init(st);
    if (active) pol.begin_row(m.dest, 0);
    for (int base = 0; base < m.len; base += 32) {
      int32_t idx_n = 0;   // the next chunk's ids, in flight while this one's rows are
      float w_n = 1.f;
      if (base + 32 + lane < m.len) {
        idx_n = p.indices ? __ldg(p.indices + m.j0 + base + 32 + lane) : m.j0 + base + 32 + lane;
        if (p.weights) w_n = __ldg(p.weights + m.j0 + base + 32 + lane);
      }
      const int cnt = m.len - base < 32 ? m.len - base : 32;
      for (int k0 = 0; k0 < cnt; k0 += SL * U) {
        typename Slice::Raw v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = k0 + u * SL + slot;
          const uint32_t src = (uint32_t)__shfl_sync(0xffffffffu, idx, e & 31);
          if (e < cnt && active) v[u] = Slice::load(my_src + (uint64_t)src * p.src_pitch);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = k0 + u * SL + slot;
          const float we = __shfl_sync(0xffffffffu, w, e & 31);
          if (e < cnt) pol.edge(st, v[u], we, 0.f);
        }
      }
      idx = idx_n; w = w_n;
    }
    auto fold = [&]() {
#pragma unroll
      for (int o = 16; o >= LPR; o >>= 1) {
        float other[NS];
#pragma unroll
        for (int k = 0; k < NS; ++k) other[k] = __shfl_xor_sync(0xffffffffu, st[k], o);
        pol.merge(st, other);   // only slot 0 is read afterwards, and there st is always the lower slot
      }
    };
    fold();
    if (slot == 0 && active) pol.end_row(st, m.dest, 0, m.len);
    if (m.dest < 0) {
      int k;
      if (last_piece(q, ~m.dest, lane, k)) {   // fold the vertex's pieces: every slot a share of them, a slice per lane, then the slots
        const int p0 = (int)__ldg(q.piece_ptr + k), p1 = (int)__ldg(q.piece_ptr + k + 1);
        pol.init(st);
        if (active)
          for (int g = p0 + slot; g < p1; g += SL) {
            float x[NS];
            const float4 *row = reinterpret_cast<const float4 *>(pol.partials + (int64_t)g * pol.dim + pol.col);
#pragma unroll
            for (int k4 = 0; k4 < NS; k4 += 4) {
              const float4 y = __ldcg(row + k4 / 4);
              x[k4] = y.x; x[k4 + 1] = y.y; x[k4 + 2] = y.z; x[k4 + 3] = y.w;
            }
            pol.merge(st, x);
          }
        fold();
        if (slot == 0 && active) {
          const int64_t v = __ldg(q.long_owners + k);
          const int64_t deg = __ldg(shadow_indptr + __ldg(owner_indptr + v + 1)) - __ldg(shadow_indptr + __ldg(owner_indptr + v));
          pol.begin_row((int32_t)v, 0);
          pol.end_row(st, (int32_t)v, 0, deg);
        }
      }
    }
  });
}

template <typename T, int RED>
it_status launch_small(const it_gather_args &a, StreamParams sp, cudaStream_t st) {
  const it_graph *g = a.g;
  using Policy = SmallPolicy<T, RED>;
  Policy pol;
  static_cast<SagePolicy<T, 16, RED, true> &>(pol) = make_policy<T, 16, RED, true>(a);
  const int slices = a.dim * (int)sizeof(T) / 16;
  const double row_bytes = (double)a.dim * sizeof(T);
  const double bytes = (double)g->e * ((a.per_edge_rows ? 0.0 : 4.0) + (a.use_edge_weights ? 4.0 : 0.0) + row_bytes) +
                       (double)g->n * (16.0 + row_bytes + (a.epi == IT_EPI_ADD_ACT ? row_bytes : 0.0));
  sp.slices = slices;
  sp.weights = a.use_edge_weights ? sp.weights : nullptr;
  if (!a.zeroed && g->n_long > 0) IT_CUDA_TRY(cudaMemsetAsync(it_done_words(a.counters), 0, (size_t)g->n_long * sizeof(int), st));
  auto go = [&]<int LPR>() -> it_status {
    const SmallShare sh = small_share(g, LPR, LPR <= 16, a.per_edge_rows && LPR >= 8 ? 5 : 8);   // (a row of 512 bytes takes the warp either way: 100k vertices / 1.6M edges 191 us, by groups 197)
    // The kernel starts early, on SMs split for the product's shared memory, and without a preference it ran with the little L1 that
    // leaves, or not, by the sizes around it: fp32 max 128-32-48-32, 31k vertices / 246k edges 109 or 120 us, now 111; bf16 mean 768-256-64,
    // 30k / 600k with hubs 177 -> 157, fp32 max 64-128-96-64, 43k / 404k 212 -> 189.  Half is what three blocks' staging takes (none: 10k / 100k
    // 35.5 -> 42.5); rows of 512 bytes stage nothing (half: fp32 max 768-256-64, 100k / 1.8M 4266 instead of 4166).  Launched plainly: 10k / 100k 37.2.
    static std::atomic<uint64_t> split{0};
    IT_TRY(split_l1(gather_small_kernel<T, LPR, Policy>, LPR <= 16 ? 50 : 0, split));
    IT_LAUNCH(IT_K_GATHER_SMALL, bytes, 0, st,
              IT_CUDA_TRY(it_launch_pdl(gather_small_kernel<T, LPR, Policy>, dim3(sh.blocks), dim3(THREADS), sh.short_blocks ? SHORT_STAGE_BYTES : 0, st, sp, pol,
                                        piece_params(g, it_done_words(a.counters)), sh, (const int64_t *)g->owner_indptr, (const int64_t *)g->shadow_indptr)));
    return IT_OK;
  };
  if (slices <= 1) return go.template operator()<1>();
  if (slices <= 2) return go.template operator()<2>();
  if (slices <= 4) return go.template operator()<4>();
  if (slices <= 8) return go.template operator()<8>();
  if (slices <= 16) return go.template operator()<16>();
  return go.template operator()<32>();
}

// ----------------------------------------------------------------------------- dispatch
template <typename T, int SB, int LPR, int RED, bool WEIGHTED>
it_status launch_policy(const it_gather_args &a, StreamParams sp, cudaStream_t st) {
  const auto pol = make_policy<T, SB, RED, WEIGHTED>(a);
  const it_graph *g = a.g;
  // algorithmic bytes: per edge the index, the optional weight and one source row; per row its
  // metadata and one output row (plus the self row it is added to)
  const double row_bytes = (double)a.dim * sizeof(T);
  auto bytes_of = [=](int b, int64_t rows) {
    return (double)g->h_list_edges[b] * ((a.per_edge_rows ? 0.0 : 4.0) + (WEIGHTED ? 4.0 : 0.0) + row_bytes) +
           (double)rows * (16.0 + row_bytes + (a.epi == IT_EPI_ADD_ACT ? row_bytes : 0.0));
  };
  auto launch = [&]<bool PAD>() {
    return launch_buckets<T, SB, LPR, PAD>(g, sp, pol, bytes_of, IT_K_GATHER_FLAT, IT_K_GATHER_EMPTY, a.counters, st);
  };
  if (a.dim * (int)sizeof(T) != SB * LPR) return launch.template operator()<true>();
  return launch.template operator()<false>();
}

template <typename T>
it_status launch_lpr(const it_gather_args &a, StreamParams sp, bool *folded, cudaStream_t st) {
  // (rows of 80 to 128 bytes cost the one kernel more than the kernels by list from about a million edges on: 60k vertices, 1M
  // edges, two layers 130 against 137 us, 130k vertices, 1.3M edges 191 against 165)
  const int row_bytes = a.dim * (int)sizeof(T);
  if (it_small_graph(a.g) && (a.partials || a.g->n_long == 0) && (row_bytes <= 64 || row_bytes > 128 || a.g->e + 6 * a.g->n <= 1400000)) {
    *folded = true;
    if (a.op == IT_GATHER_MAX) return launch_small<T, RED_MAX>(a, sp, st);
    if (a.op == IT_GATHER_MIN) return launch_small<T, RED_MIN>(a, sp, st);
    return launch_small<T, RED_SUM>(a, sp, st);
  }
  const bool w = a.use_edge_weights != 0;
  return dispatch_wide_rows(row_bytes, [&]<int SB, int LPR>() {
    if (a.op == IT_GATHER_MAX) return w ? launch_policy<T, SB, LPR, RED_MAX, true>(a, sp, st) : launch_policy<T, SB, LPR, RED_MAX, false>(a, sp, st);
    if (a.op == IT_GATHER_MIN) return w ? launch_policy<T, SB, LPR, RED_MIN, true>(a, sp, st) : launch_policy<T, SB, LPR, RED_MIN, false>(a, sp, st);
    return w ? launch_policy<T, SB, LPR, RED_SUM, true>(a, sp, st) : launch_policy<T, SB, LPR, RED_SUM, false>(a, sp, st);
  });
}

}  // namespace
