// Gather: the aggregate over the in-edges of one shadow row (sum / mean / max / min of w_e * h_src).  The edge streaming
// itself lives in stream.cuh; this file supplies the per-lane state and what happens at the end of a row.  Included by
// one source file per storage type (the kernels are many; they compile side by side).
#pragma once
#include "stream.cuh"

namespace {

using namespace it_stream;

// Per lane: VEC fp32 accumulators for its slice of the row.

template <typename T, int SB, int RED, bool WEIGHTED_>
struct SagePolicy {
  using Slice = RowSlice<T, SB>;
  static constexpr int VEC = Slice::VEC;
  static constexpr int NS = VEC;
  static constexpr bool WEIGHTED = WEIGHTED_, HAS_EXTRA = false, NEEDS_OWNER = false;
  float *__restrict__ partials;
  void *__restrict__ dst;
  const void *__restrict__ self_term;
  const float *__restrict__ bias;
  int dim, dst_ld, self_ld, is_mean, epi, act;   // dim: width of this column chunk; *_ld: row lengths of dst / the self term
  // per-thread
  int col;
  float self[VEC];

  void empty_rows(it_empty_rows_args &a) const {
    const bool raw = epi == IT_EPI_RAW_F32;
    a.kind = epi == IT_EPI_ADD_ACT ? IT_EMPTY_SELF : (epi == IT_EPI_BIAS_ACT ? IT_EMPTY_BIAS : IT_EMPTY_VALUE);
    a.dst = dst; a.dim = dim; a.dtype = raw || sizeof(T) == 4 ? IT_F32 : IT_BF16; a.pitch = (int64_t)dst_ld * (raw ? 4 : (int)sizeof(T));
    a.self = self_term; a.self_pitch = (int64_t)self_ld * (int)sizeof(T);
    a.value = raw ? (RED == RED_MAX ? -INFINITY : (RED == RED_MIN ? INFINITY : 0.f)) : 0.f;
    a.bias = bias; a.act = (it_act)act;
  }
  __device__ __forceinline__ void setup(int t) { col = t * VEC; }
  __device__ __forceinline__ void init(float (&st)[NS]) const {
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
#pragma unroll
    for (int k = 0; k < NS; ++k) st[k] = RED == RED_MAX ? fmaxf(st[k], o[k]) : (RED == RED_MIN ? fminf(st[k], o[k]) : st[k] + o[k]);
  }
  // the matching slice of the self term is fetched when the row starts, so that end_row does not wait for it
  __device__ __forceinline__ void begin_row(int32_t dest, int32_t) {
    if (epi == IT_EPI_ADD_ACT && dest >= 0)
      Slice::unpack(Slice::load_stream(reinterpret_cast<const char *>(self_term) + ((int64_t)dest * self_ld + col) * (int64_t)sizeof(T)), self);
  }
  __device__ __forceinline__ void end_row(float (&st)[NS], int32_t dest, int32_t, int64_t len) const {
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

// ----------------------------------------------------------------------------- dispatch
template <typename T, int SB, int LPR, int RED, bool WEIGHTED>
it_status launch_policy(const it_gather_args &a, StreamParams sp, int64_t bound_lo, int64_t bound_hi, cudaStream_t st) {
  SagePolicy<T, SB, RED, WEIGHTED> pol;
  pol.partials = a.partials; pol.dst = a.dst; pol.self_term = a.self_term; pol.bias = a.bias; pol.dim = a.dim; pol.dst_ld = a.dst_ld > 0 ? a.dst_ld : a.dim; pol.self_ld = a.self_ld > 0 ? a.self_ld : a.dim;
  pol.is_mean = a.op == IT_GATHER_MEAN && a.epi != IT_EPI_RAW_F32; pol.epi = a.epi; pol.act = a.act; pol.col = 0;
  const it_graph *g = a.g;
  // algorithmic bytes: per edge the index, the optional weight and one source row; per row its
  // metadata and one output row (plus the self row it is added to)
  const double row_bytes = (double)a.dim * sizeof(T);
  auto bytes_of = [=](int b, int64_t rows) {
    return (double)g->h_list_edges[b] * ((a.per_edge_rows ? 0.0 : 4.0) + (WEIGHTED ? 4.0 : 0.0) + row_bytes) +
           (double)rows * (16.0 + row_bytes + (a.epi == IT_EPI_ADD_ACT ? row_bytes : 0.0));
  };
  auto launch = [&]<bool PAD>() {
    return launch_buckets<T, SB, LPR, PAD>(g, sp, pol, bytes_of, IT_K_GATHER_FLAT, IT_K_GATHER_EMPTY, bound_lo, bound_hi, a.counters, st);
  };
  if constexpr (SB == 16) {
    if (a.dim * (int)sizeof(T) != SB * LPR) return launch.template operator()<true>();
  }
  return launch.template operator()<false>();
}

template <typename T>
it_status launch_lpr(const it_gather_args &a, StreamParams sp, cudaStream_t st) {
  const bool w = a.use_edge_weights != 0;
  return dispatch_row_bytes(a.dim * (int)sizeof(T), true, [&]<int SB, int LPR>(int64_t lo, int64_t hi) {
    if (a.op == IT_GATHER_MAX) return w ? launch_policy<T, SB, LPR, RED_MAX, true>(a, sp, lo, hi, st) : launch_policy<T, SB, LPR, RED_MAX, false>(a, sp, lo, hi, st);
    if (a.op == IT_GATHER_MIN) return w ? launch_policy<T, SB, LPR, RED_MIN, true>(a, sp, lo, hi, st) : launch_policy<T, SB, LPR, RED_MIN, false>(a, sp, lo, hi, st);
    return w ? launch_policy<T, SB, LPR, RED_SUM, true>(a, sp, lo, hi, st) : launch_policy<T, SB, LPR, RED_SUM, false>(a, sp, lo, hi, st);
  });
}

}  // namespace
