// The GAT reduce with the attention weights of many edges computed at once, for rows of 64 to 512 bytes in 16-byte
// slices (bf16 128 or fp32 64 columns: 256 bytes) and 1, 2, 4 or 8 heads.
//
// The running-softmax policy of gat.cu works edge by edge: every lane of a row recomputes the logit and the exponential
// of its head and rescales its accumulators at each edge, about 35 instructions per edge and slice, which kept the
// kernels at 72-79 % of their issue slots with DRAM half idle.  Here a step covers E edges at once (32 of a warp's row, 8 of a
// lane group's): the (edge, head) pairs are spread over the lanes, one maximum per head and step is taken by
// shuffles, each pair's weight exp(e - m) is computed once, accumulators are rescaled once per step, and an edge then
// costs its slice's multiply-adds.  The state is the same (max, sum, weighted accumulator), so partial states of split
// vertices merge as before.  Measured on 1.25M vertices, 25M edges, bf16 4 heads of 32 (256-byte rows), before -> after: rows
// of at most 8 edges 252 -> 194 us, 9..32 edges 188 -> 157, 33..1024 edges 435 -> 418, longer 441 -> 400 (DRAM at 0.8 of its
// peak, as a copy reaches); with edge features in the logits the source rows are no longer copied in edge order (8M edges,
// fp32 64 columns: 1.61 -> 0.83 ms for the layer).
//
// Included by gat.cu.
#pragma once

#include "gather_small.cuh"

namespace {

using namespace it_stream;

struct GatParams {
  const float *__restrict__ scores;       // source-side logit term: [n_src, H], or [n_edges, H] when per_edge (rows of `stride`)
  const float *__restrict__ scores_dst;   // [local destinations, 2H]: destination scores in the second half
  int stride;                             // floats from one row of it to the next (H, or 2H for the interleaved score rows)
  int per_edge;                           // the term belongs to the edge (edge features in the logits), not to its source
  float slope;
  int head_dim;
};

// Accumulators of one slice plus the sum of the weights.  All states of one warp's row share their maximum, so folding
// slots is a plain sum.
template <typename T>
struct GatAcc {
  using Slice = RowSlice<T, 16>;
  static constexpr int VEC = Slice::VEC, NS = VEC + 1;
  static constexpr bool HAS_EXTRA = false, WEIGHTED = false;
  __device__ __forceinline__ const float *extra_ptr(uint32_t) const { return nullptr; }
  __device__ __forceinline__ void init(float (&st)[NS]) const {
#pragma unroll
    for (int k = 0; k < NS; ++k) st[k] = 0.f;
  }
  __device__ __forceinline__ void edge(float (&st)[NS], const uint4 &raw, float w) const {
    float f[VEC];
    Slice::unpack(raw, f);
#pragma unroll
    for (int k = 0; k < VEC; k += 2) fma_f32x2(st[k], st[k + 1], w, f[k], f[k + 1]);
    st[VEC] += w;
  }
  __device__ __forceinline__ void scale(float (&st)[NS], float s) const {
#pragma unroll
    for (int k = 0; k < NS; ++k) st[k] *= s;
  }
  __device__ __forceinline__ void merge(float (&st)[NS], const float (&o)[NS]) const {
#pragma unroll
    for (int k = 0; k < NS; ++k) st[k] += o[k];
  }
};

// The bias in shared memory, for the end of a row (its address need not be 16-byte aligned in global memory).
template <class Policy>
__device__ __forceinline__ void stage_bias(Policy &pol, float (&buf)[256]) {
  for (int i = threadIdx.x; i < pol.dim; i += THREADS) buf[i] = pol.bias ? pol.bias[i] : 0.f;
  __syncthreads();
  pol.bias_s = (uint32_t)__cvta_generic_to_shared(&buf[0]);
}

__device__ __forceinline__ float leaky(float x, float slope) { return x > 0.f ? x : slope * x; }

// ----------------------------------------------------------------------------- one warp per row (or per part of a row)
// Lane = (edge el = lane / H, head hl = lane % H) for the logits; pair i of a lane is edge el + i * 32 / H of the chunk.
template <typename T, int LPR, int H>
struct GatPairs {
  static constexpr int EP = 32 / H;   // edges covered by one pair per lane
  const StreamParams &p;
  const GatParams &q;
  const int lane, hl, el, hc;         // hc: head of the lane's slice
  const uint32_t pw;                  // shared-window address of this warp's weights [32][H]
  float x_c[H], x_n[H];               // logit terms of the current / the next chunk
  float sd_c, sd_n;                   // destination scores of their rows
  float m;                            // running maximum of head hl
  GatAcc<T> acc;
  float st[GatAcc<T>::NS];

  __device__ __forceinline__ GatPairs(const StreamParams &p_, const GatParams &q_, int lane_, uint32_t pw_)
      : p(p_), q(q_), lane(lane_), hl(lane_ % H), el(lane_ / H), hc((lane_ % LPR) * GatAcc<T>::VEC / q_.head_dim), pw(pw_) {
    sd_c = sd_n = 0.f; m = -INFINITY;
#pragma unroll
    for (int i = 0; i < H; ++i) x_c[i] = x_n[i] = 0.f;
    acc.init(st);
  }
  // the ids of chunk c have landed: fetch its logit terms (into the "next" registers)
  __device__ __forceinline__ void ahead(const Chunk &c) {
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const int e = el + i * EP;
      const uint32_t s = (uint32_t)__shfl_sync(0xffffffffu, c.idx, e);
      if (e < c.cnt) x_n[i] = __ldg(q.scores + (q.per_edge ? (uint64_t)(c.j + e) : (uint64_t)s) * q.stride + hl);
    }
    sd_n = __ldg(q.scores_dst + (int64_t)c.owner * (2 * H) + H + hl);
  }
  // chunk c becomes the current one: its attention weights
  __device__ __forceinline__ void begin(const Chunk &c, bool first) {
    sd_c = sd_n;
    float mr = -INFINITY;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      x_c[i] = el + i * EP < c.cnt ? leaky(x_n[i] + sd_c, q.slope) : -INFINITY;
      mr = fmaxf(mr, x_c[i]);
    }
#pragma unroll
    for (int o = H; o < 32; o <<= 1) mr = fmaxf(mr, __shfl_xor_sync(0xffffffffu, mr, o));
    if (first) { m = -INFINITY; acc.init(st); }
    const float m_new = fmaxf(m, mr);
    const float s = __shfl_sync(0xffffffffu, it_exp(m - m_new), hc);   // exp(-inf) = 0 for the first chunk of a row
    if (!first) acc.scale(st, s);
    m = m_new;
    __syncwarp();   // the previous chunk's weights have been read
#pragma unroll
    for (int i = 0; i < H; ++i)
      asm volatile("st.shared.f32 [%0], %1;" ::"r"(pw + (uint32_t)((lane + 32 * i) * 4)), "f"(it_exp(x_c[i] - m)) : "memory");
    __syncwarp();
  }
  __device__ __forceinline__ void clear() { m = -INFINITY; acc.init(st); }
  __device__ __forceinline__ float maximum() const { return __shfl_sync(0xffffffffu, m, hc); }   // of the slice's head
  __device__ __forceinline__ float weight(int k) const { return lds_f32(pw + (uint32_t)((k * H + hc) * 4)); }
};

// The largest x of the warp (of numbers: a NaN is no candidate).
__device__ __forceinline__ float warp_max(float x) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(x));
  return r;
}
// H consecutive floats, aligned to H of them (at most 16 bytes)
template <int H>
__device__ __forceinline__ void load_heads(const float *p, float (&x)[H]) {
  if constexpr (H == 1) x[0] = __ldg(p);
  else if constexpr (H == 2) { const float2 v = __ldg(reinterpret_cast<const float2 *>(p)); x[0] = v.x; x[1] = v.y; }
  else {
#pragma unroll
    for (int i = 0; i < H; i += 4) {
      const float4 v = __ldg(reinterpret_cast<const float4 *>(p + i));
      x[i] = v.x; x[i + 1] = v.y; x[i + 2] = v.z; x[i + 3] = v.w;
    }
  }
}
template <int H>
__device__ __forceinline__ float pick(const float (&x)[H], int h) {   // x[h], h not known at compile time
  float r = x[0];
#pragma unroll
  for (int i = 1; i < H; ++i) r = h == i ? x[i] : r;
  return r;
}

// Lane = edge of the chunk, with all its heads: one load of its logit terms and one warp reduction per head, where a lane per pair of
// edge and head takes a load, an id shuffle and a store per head.
template <typename T, int LPR, int H>
struct GatEdges {
  const StreamParams &p;
  const GatParams &q;
  const int lane, hc;                 // hc: head of the lane's slice
  const uint32_t pw;                  // shared-window address of this warp's weights [32][H]
  float x_n[H], sd_n[H];              // of the next chunk: logit terms, destination scores of its row
  float m[H];                         // running maxima
  GatAcc<T> acc;
  float st[GatAcc<T>::NS];

  __device__ __forceinline__ GatEdges(const StreamParams &p_, const GatParams &q_, int lane_, uint32_t pw_)
      : p(p_), q(q_), lane(lane_), hc((lane_ % LPR) * GatAcc<T>::VEC / q_.head_dim), pw(pw_) {
#pragma unroll
    for (int i = 0; i < H; ++i) { x_n[i] = sd_n[i] = 0.f; m[i] = -INFINITY; }
    acc.init(st);
  }
  // the ids of chunk c have landed: fetch its logit terms (into the "next" registers)
  __device__ __forceinline__ void ahead(const Chunk &c) {
    if (lane < c.cnt) load_heads<H>(q.scores + (q.per_edge ? (uint64_t)(c.j + lane) : (uint64_t)(uint32_t)c.idx) * q.stride, x_n);
    load_heads<H>(q.scores_dst + (int64_t)c.owner * (2 * H) + H, sd_n);
  }
  // chunk c becomes the current one: its attention weights
  __device__ __forceinline__ void begin(const Chunk &c, bool first) {
    float x[H], s[H];
    if (first) acc.init(st);
#pragma unroll
    for (int i = 0; i < H; ++i) {
      x[i] = lane < c.cnt ? leaky(x_n[i] + sd_n[i], q.slope) : -INFINITY;
      const float was = first ? -INFINITY : m[i];
      m[i] = fmaxf(was, warp_max(x[i]));
      s[i] = it_exp(was - m[i]);   // exp(-inf) = 0 for the first chunk of a row
      x[i] = it_exp(x[i] - m[i]);
    }
    if (!first) acc.scale(st, pick<H>(s, hc));
    __syncwarp();   // the previous chunk's weights have been read
    const uint32_t at = pw + (uint32_t)(lane * H * 4);
    if constexpr (H == 1) asm volatile("st.shared.f32 [%0], %1;" ::"r"(at), "f"(x[0]) : "memory");
    else if constexpr (H == 2) asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(at), "f"(x[0]), "f"(x[1]) : "memory");
    else {
#pragma unroll
      for (int i = 0; i < H; i += 4)
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at + i * 4), "f"(x[i]), "f"(x[i + 1]), "f"(x[i + 2]), "f"(x[i + 3]) : "memory");
    }
    __syncwarp();
  }
  __device__ __forceinline__ float weight(int k) const { return lds_f32(pw + (uint32_t)((k * H + hc) * 4)); }
  __device__ __forceinline__ float maximum() const { return pick<H>(m, hc); }   // of the slice's head
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < H; ++i) m[i] = -INFINITY;
    acc.init(st);
  }
};
// Which of the two: the registers of eight heads spill, and so do those of bf16 rows in the chunk kernel, whose accumulators are twice
// as many (5M vertices / 100M edges, 4 heads: pairs 10.8 ms, edges 11.3; fp32 4 heads of 16, 500k / 8M with edge features: pairs 572 us,
// edges 533).  In the kernel for small graphs 30k / 420k, bf16 4 heads: pairs 65 us, edges 63.
template <typename T, int LPR, int H> using GatWarp = std::conditional_t<sizeof(T) == 4 && H <= 4, GatEdges<T, LPR, H>, GatPairs<T, LPR, H>>;
template <typename T, int LPR, int H> using GatSmallWarp = std::conditional_t<H <= 4, GatEdges<T, LPR, H>, GatPairs<T, LPR, H>>;

#ifndef IT_GAT_CHUNK_BLOCKS
#define IT_GAT_CHUNK_BLOCKS 3   // resident CTAs per SM: at four the 64 registers a thread gets spill (measured: 3 to 5 % more time)
#endif
#ifndef IT_GAT_STAGE_ROWS
#define IT_GAT_STAGE_ROWS 8   // 512-byte groups of rows per stage of the chunk kernel's ring (4: 2.5 % more time on 5M vertices / 100M edges)
#endif
// (64-byte rows: 32 edges are four groups)
template <int LPR> constexpr int gat_stage_rows() { return LPR == 4 ? 4 : IT_GAT_STAGE_ROWS; }
template <int LPR, int H> constexpr int gat_bytes_per_warp() { return ring_bytes_per_warp<16, false, gat_stage_rows<LPR>()>() + 32 * H * 4; }

template <typename T, int LPR, int H>
__global__ void __launch_bounds__(THREADS, IT_GAT_CHUNK_BLOCKS) gat_rows_chunk_kernel(StreamParams p, GatParams q, GatPolicy<T, 16> pol) {
  extern __shared__ uint4 ring_raw[];
  static_assert(gat_bytes_per_warp<LPR, H>() % 16 == 0, "a warp's weights are written 16 bytes at a time");
  const int lane = threadIdx.x & 31;
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(ring_raw) + (uint32_t)(threadIdx.x >> 5) * (uint32_t)gat_bytes_per_warp<LPR, H>();
  RingWarp<T, 16, LPR, GatAcc<T>, false, gat_stage_rows<LPR>()> rw;
  rw.setup(base, p.src, p.src_pitch, p.slices, lane);
  pol.setup(lane % LPR);
  __shared__ __align__(16) float bias_buf[256];   // (read 16 bytes at a time)
  stage_bias(pol, bias_buf);
  GatWarp<T, LPR, H> gw(p, q, lane, base + ring_bytes_per_warp<16, false, gat_stage_rows<LPR>()>());
  ChunkCursor<false, true> cur(p, lane);
  chunk_walk<LPR, true>(rw, gw.acc, cur, [&](Chunk &c) { gw.ahead(c); }, [&](const Chunk &c, bool first) { gw.begin(c, first); },
      [&](int k, const uint4 &raw, bool valid) {
        const float w = gw.weight(k);
        if (valid) gw.acc.edge(gw.st, raw, w);
      },
      [&](const Chunk &c) {
        rw.fold(gw.acc, gw.st);
        const float mh = gw.maximum();
        float full[GatPolicy<T, 16>::NS];
#pragma unroll
        for (int k = 0; k < GatAcc<T>::VEC; ++k) full[k] = gw.st[k];
        full[GatAcc<T>::VEC] = mh;
        full[GatAcc<T>::VEC + 1] = gw.st[GatAcc<T>::VEC];
        if (rw.slot == 0) pol.end_row(full, c.dest, 0, 0);
      });
}

// ----------------------------------------------------------------------------- short rows: one lane group each
// Rows of at most a few dozen edges, up to 256 bytes each: a group of LPR lanes owns a row and walks it in rounds of up
// to E = 8 edges (4 for 64-byte rows); the groups of a warp run in lockstep, a round as long as its longest row.  While the rows of one round are
// reduced, the source rows and logit terms of the next round are in flight (two staging buffers in shared memory), the ids
// of the round after it, and the records of the rows after that.
#ifndef IT_GAT_SHORT_BLOCKS
#define IT_GAT_SHORT_BLOCKS 3   // resident CTAs per SM: 64 KB of staging each
#endif
// block / blocks: which share of the rows p.row_lo .. p.row_hi this block walks; short_buf: [2][E][THREADS] in shared memory.
template <typename T, int LPR, int H>
__device__ __forceinline__ void gat_short_rows(const StreamParams &p, const GatParams &q, const GatPolicy<T, 16> &pol, int block, int blocks, uint4 *short_buf) {
  using Acc = GatAcc<T>;
  constexpr int E = LPR < IT_SHORT_EDGES ? LPR : IT_SHORT_EDGES;
  constexpr int EP = LPR / H;                            // edges covered by one pair per lane
  constexpr int PP = E > EP ? E / EP : 1;                // (edge, head) pairs per lane
  static_assert(H <= LPR && E <= LPR, "a group holds its pairs and its ids");
  const int lane = threadIdx.x & 31, t = lane % LPR, gbase = lane - t;
  const int hl = t % H, el = t / H;
  const int hc = t * Acc::VEC / q.head_dim;              // head of the lane's slice
  const char *my_src = reinterpret_cast<const char *>(p.src) + (size_t)t * 16;
  const uint32_t ROWB = p.src_pitch;
  constexpr uint32_t SLOT = THREADS * 16, BUF = E * SLOT;
  uint32_t buf = (uint32_t)__cvta_generic_to_shared(short_buf + threadIdx.x), other = buf + BUF;
  const int64_t sweep = (int64_t)blocks * (THREADS / LPR);

  struct Row { int64_t j0; int len, most, dest, owner; float sd; };   // most: longest row of the warp's groups (0: no rows left)
  auto load_row = [&](int64_t i0, Row &r) {
    r.j0 = 0; r.len = 0; r.dest = 0; r.owner = 0;
    const int64_t i = i0 + lane / LPR;
    if (i < p.row_hi) {
      const it_row_meta m = load_meta(p.meta + i);
      r.j0 = m.j0; r.len = m.len; r.dest = m.dest;
      r.owner = __ldcs(p.owner + i);
    }
  };
  auto finish_row = [&](Row &r) {   // the record has landed: what hangs on it
    r.most = __reduce_max_sync(0xffffffffu, r.len);
    r.sd = __ldg(q.scores_dst + (int64_t)r.owner * (2 * H) + H + hl);   // owner 0 for a missing row: read, not used
  };
  auto load_ids = [&](const Row &r, int k) -> int32_t {
    if (t < E && k + t < r.len) return p.indices ? __ldcs(p.indices + r.j0 + k + t) : (int32_t)(r.j0 + k + t);
    return 0;
  };
  // the source rows and logit terms of edges [k, k + E) of row r, whose ids are in idx
  auto issue = [&](const Row &r, int k, int32_t idx, uint32_t d, float (&x)[PP]) {
#pragma unroll
    for (int u = 0; u < E; ++u) {
      if (k + u >= r.most) break;   // warp-uniform
      const uint32_t s = (uint32_t)__shfl_sync(0xffffffffu, idx, gbase + u);
      if (k + u < r.len) cp_async_slice<16>(d + (uint32_t)u * SLOT, my_src + (uint64_t)s * ROWB);
    }
    cp_async_commit();
#pragma unroll
    for (int u = 0; u < PP; ++u) {
      const int e = el + u * EP;
      const uint32_t s = (uint32_t)__shfl_sync(0xffffffffu, idx, gbase + (e & (E - 1)));
      x[u] = __int_as_float(0x7fffffff);   // NaN stays NaN whatever the slope; the weight of a pair without an edge is not used
      if (e < E && k + e < r.len) x[u] = __ldg(q.scores + (q.per_edge ? (uint64_t)(r.j0 + k + e) : (uint64_t)s) * q.stride + hl);
    }
  };

  int64_t i0 = p.row_lo + (int64_t)block * (THREADS / LPR) + (threadIdx.x >> 5) * (32 / LPR);   // warp-uniform
  Row r0, r1, r2;
  load_row(i0, r0); load_row(i0 + sweep, r1); load_row(i0 + 2 * sweep, r2);
  finish_row(r0);
  if (r0.most == 0) return;   // warp-uniform
  finish_row(r1);
  float x_a[PP], x_b[PP];
  int32_t idx_b = load_ids(r0, 0);
  issue(r0, 0, idx_b, buf, x_a);
  idx_b = r0.most > E ? load_ids(r0, E) : load_ids(r1, 0);
  Acc acc;
  float st[Acc::NS];
  for (; r0.most > 0; i0 += sweep) {
    Row r3;
    load_row(i0 + 3 * sweep, r3);
    finish_row(r2);
    float m = -INFINITY;
    acc.init(st);
    for (int k0 = 0; k0 < r0.most; k0 += E) {
      // the next round, and the ids of the one after it
      if (k0 + E < r0.most) issue(r0, k0 + E, idx_b, other, x_b);
      else issue(r1, 0, idx_b, other, x_b);
      if (k0 + 2 * E < r0.most) idx_b = load_ids(r0, k0 + 2 * E);
      else if (k0 + E < r0.most) idx_b = load_ids(r1, 0);
      else idx_b = r1.most > E ? load_ids(r1, E) : load_ids(r2, 0);
      // this round: the weights ...
      float mr = -INFINITY;
#pragma unroll
      for (int u = 0; u < PP; ++u) {
        x_a[u] = leaky(x_a[u] + r0.sd, q.slope);
        mr = fmaxf(mr, x_a[u]);   // (of a NaN and a number the number: pairs without an edge do not count)
      }
#pragma unroll
      for (int o = H; o < LPR; o <<= 1) mr = fmaxf(mr, __shfl_xor_sync(0xffffffffu, mr, o));
      const float m_new = fmaxf(m, mr);
      if (k0 > 0) {   // rows whose edges are used up: m_new = m, a factor of 1
        const float s = __shfl_sync(0xffffffffu, it_exp(m - m_new), gbase + hc);
        acc.scale(st, s);
      }
      m = m_new;
#pragma unroll
      for (int u = 0; u < PP; ++u) x_a[u] = it_exp(x_a[u] - m);
      // ... and the slices
      cp_async_wait<1>();
#pragma unroll
      for (int u = 0; u < E; ++u) {
        if (k0 + u >= r0.most) break;
        const float w = __shfl_sync(0xffffffffu, x_a[u / EP], gbase + (u % EP) * H + hc);
        if (k0 + u < r0.len) acc.edge(st, lds_slice<16>(buf + (uint32_t)u * SLOT), w);
      }
#pragma unroll
      for (int u = 0; u < PP; ++u) x_a[u] = x_b[u];
      const uint32_t sw = buf; buf = other; other = sw;
    }
    const float mh = __shfl_sync(0xffffffffu, m, gbase + hc);
    if (r0.len > 0) {
      float full[GatPolicy<T, 16>::NS];
#pragma unroll
      for (int k = 0; k < Acc::VEC; ++k) full[k] = st[k];
      full[Acc::VEC] = mh;
      full[Acc::VEC + 1] = st[Acc::VEC];
      pol.end_row(full, r0.dest, 0, 0);
    }
    r0 = r1; r1 = r2; r2 = r3;
  }
  cp_async_wait<0>();
}
template <typename T, int LPR, int H>
__global__ void __launch_bounds__(THREADS, IT_GAT_SHORT_BLOCKS) gat_short_rows_kernel(StreamParams p, GatParams q, GatPolicy<T, 16> pol) {
  extern __shared__ uint4 short_buf[];
  __shared__ __align__(16) float bias_buf[256];   // (read 16 bytes at a time)
  pol.setup(threadIdx.x % LPR);
  stage_bias(pol, bias_buf);
  gat_short_rows<T, LPR, H>(p, q, pol, blockIdx.x, gridDim.x, short_buf);
}

// ----------------------------------------------------------------------------- small graphs: every list of a layer in one kernel
template <typename T, int LPR, int H>
__global__ void __launch_bounds__(THREADS, SMALL_BLOCKS) gat_small_kernel(StreamParams p, GatParams q, GatPolicy<T, 16> pol, PieceParams pq, SmallShare sh) {
  constexpr int SL = 32 / LPR, U = 4, VEC = GatAcc<T>::VEC, NS = GatPolicy<T, 16>::NS;   // U rows in flight per lane
  extern __shared__ uint4 short_buf[];
  __shared__ __align__(16) float weights[THREADS / 32][32 * H];
  __shared__ __align__(16) float bias_buf[256];   // (read 16 bytes at a time)
  it_allow_next();
  const int lane = threadIdx.x & 31, slot = lane / LPR, t = lane % LPR;
  pol.setup(t);
  const char *my_src = reinterpret_cast<const char *>(p.src) + (size_t)t * 16;
  stage_bias(pol, bias_buf);
  if ((int)blockIdx.x < sh.short_blocks) {
    p.row_lo = sh.short_lo; p.row_hi = sh.short_hi;
    gat_short_rows<T, LPR, H>(p, q, pol, blockIdx.x, sh.short_blocks, short_buf);
    return;
  }
  if ((int)blockIdx.x < sh.short_blocks + sh.empty_blocks) {
    float none[NS];
    pol.init(none);
    small_empties(sh, [&](int b, int n) {
      const int dest = lane < n ? __ldcs(&p.meta[b + lane].dest) : 0;
      for (int k = 0; k < n; k += SL) {
        const int d = __shfl_sync(0xffffffffu, dest, (k + slot) & 31);
        if (k + slot < n) pol.end_row(none, d, 0, 0);
      }
    });
    return;
  }
  GatSmallWarp<T, LPR, H> gw(p, q, lane, (uint32_t)__cvta_generic_to_shared(&weights[threadIdx.x >> 5][0]));
  small_walk<false, true>(p, sh, lane, [&](const SmallRow &m, int32_t idx, float) {
    gw.clear();
    for (int base = 0; base < m.len; base += 32) {
      Chunk c;
      c.cnt = m.len - base < 32 ? m.len - base : 32;
      int32_t idx_n = 0;   // the next chunk's ids, in flight while this one's rows are
      if (base + 32 + lane < m.len) idx_n = p.indices ? __ldg(p.indices + m.j0 + base + 32 + lane) : m.j0 + base + 32 + lane;
      c.idx = idx; c.owner = m.owner; c.j = m.j0 + base;
      gw.ahead(c);
      uint4 v[U];
      auto load = [&](int k0) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = k0 + u * SL + slot;
          const uint32_t s = (uint32_t)__shfl_sync(0xffffffffu, idx, e & 31);
          if (e < c.cnt) v[u] = __ldg(reinterpret_cast<const uint4 *>(my_src + (uint64_t)s * p.src_pitch));
        }
      };
      load(0);
      gw.begin(c, base == 0);
      for (int k0 = 0; k0 < c.cnt; k0 += SL * U) {
        if (k0 > 0) load(k0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = k0 + u * SL + slot;
          if (e < c.cnt) gw.acc.edge(gw.st, v[u], gw.weight(e));
        }
      }
      idx = idx_n;
    }
#pragma unroll
    for (int o = 16; o >= LPR; o >>= 1) {
      float other[GatAcc<T>::NS];
#pragma unroll
      for (int k = 0; k < GatAcc<T>::NS; ++k) other[k] = __shfl_xor_sync(0xffffffffu, gw.st[k], o);
      gw.acc.merge(gw.st, other);
    }
    const float mh = gw.maximum();
    float full[NS];
#pragma unroll
    for (int k = 0; k < VEC; ++k) full[k] = gw.st[k];
    full[VEC] = mh;
    full[VEC + 1] = gw.st[VEC];
    if (slot == 0) pol.end_row(full, m.dest, 0, m.len);
    if (m.dest < 0) {
      int k;
      if (last_piece(pq, ~m.dest, lane, k)) {   // merge the vertex's pieces: every slot a share of them, a slice per lane, then the slots
        const int p0 = (int)__ldg(pq.piece_ptr + k), p1 = (int)__ldg(pq.piece_ptr + k + 1);
        const int stride = gat_partial_stride(pol.dim, pol.heads);
        pol.init(full);
        for (int g = p0 + slot; g < p1; g += SL) {
          const float *row = pol.partials + (int64_t)g * stride;
          float x[NS];
#pragma unroll
          for (int k4 = 0; k4 < VEC; k4 += 4) {
            const float4 y = __ldcg(reinterpret_cast<const float4 *>(row + pol.col + k4));
            x[k4] = y.x; x[k4 + 1] = y.y; x[k4 + 2] = y.z; x[k4 + 3] = y.w;
          }
          x[VEC] = __ldcg(row + pol.dim + pol.head);
          x[VEC + 1] = __ldcg(row + pol.dim + pol.heads + pol.head);
          pol.merge(full, x);
        }
#pragma unroll
        for (int o = 16; o >= LPR; o >>= 1) {
          float x[NS];
#pragma unroll
          for (int k4 = 0; k4 < NS; ++k4) x[k4] = __shfl_xor_sync(0xffffffffu, full[k4], o);
          pol.merge(full, x);
        }
        if (slot == 0) pol.end_row(full, __ldg(pq.long_owners + k), 0, 1);
      }
    }
  });
}

template <typename T, int LPR, int H>
it_status launch_gat_small(const it_gat_args &a, StreamParams p, const GatPolicy<T, 16> &pol, cudaStream_t st) {
  const it_graph *g = a.g;
  GatParams q;
  q.scores = pol.scores; q.scores_dst = pol.scores_dst; q.stride = pol.src_stride; q.per_edge = a.per_edge_scores; q.slope = pol.slope; q.head_dim = pol.head_dim;
  p.slices = LPR;
  if (!a.zeroed && g->n_long > 0) IT_CUDA_TRY(cudaMemsetAsync(it_done_words(a.counters), 0, (size_t)g->n_long * sizeof(int), st));
  const double row_bytes = (double)pol.dim * sizeof(T);
  const double bytes = (double)g->e * (4.0 + 4.0 * H + row_bytes) + (double)g->n * (20.0 + 4.0 * H + row_bytes);
  const SmallShare sh = small_share(g, LPR, true, a.per_edge_scores ? 5 : 8);   // (logit terms in edge order come cheaper: 20k vertices / 300k edges 43 us, with 8 47)
  const int smem = sh.short_blocks ? 2 * IT_SHORT_EDGES * THREADS * 16 : 0;
  static std::atomic<uint64_t> configured{0};
  IT_TRY(allow_dynamic_smem(gat_small_kernel<T, LPR, H>, 2 * IT_SHORT_EDGES * THREADS * 16, configured));
  // (Not started early: on SMs split for the dense product's shared memory it finds little L1, which its score and row loads
  // live on: 30k vertices, two layers 84 us, started early 98.)
  IT_LAUNCH(IT_K_GAT_SMALL, bytes, 0, st,
            gat_small_kernel<T, LPR, H><<<sh.blocks, THREADS, smem, st>>>(p, q, pol, piece_params(g, it_done_words(a.counters)), sh));
  IT_CUDA_TRY(cudaGetLastError());
  return IT_OK;
}

// ----------------------------------------------------------------------------- launches
template <typename T, int LPR, int H, class BytesF>
it_status launch_gat_rows(const it_gat_args &a, StreamParams p, const GatPolicy<T, 16> &pol, BytesF bytes_of, cudaStream_t st) {
  const it_graph *g = a.g;
  GatParams q;
  q.scores = pol.scores; q.scores_dst = pol.scores_dst; q.stride = pol.src_stride; q.per_edge = a.per_edge_scores; q.slope = pol.slope; q.head_dim = pol.head_dim;
  p.slices = LPR;
  if (a.counters) IT_CUDA_TRY(cudaMemsetAsync(a.counters, 0, (IT_MAX_BUCKETS + 1) * sizeof(int), st));
  bool chunked = false;
  for (int b = g->n_lists - (pol.partials ? 1 : 2); b >= 0; --b) {   // (without room for partial rows no pieces are walked)
    const int64_t lo = g->h_list_offsets[b], hi = g->h_list_offsets[b + 1], bound = g->list_bounds[b];
    if (hi <= lo) continue;
    p.row_lo = lo; p.row_hi = hi;
    const int64_t rows = hi - lo;
    const double bytes = bytes_of(b, rows);
    constexpr int smem = (THREADS / 32) * gat_bytes_per_warp<LPR, H>();
    if (bound == 0) {
      it_empty_rows_args er;
      pol.empty_rows(er);
      er.g = g; er.row_lo = lo; er.row_hi = hi;
      IT_TRY(it_launch_empty_rows(er, IT_K_GAT_EMPTY, bytes, st));
    } else if (LPR <= 16 && bound <= IT_SHORT_BELOW) {
      if constexpr (LPR <= 16) {
        constexpr int sbytes = 2 * IT_SHORT_EDGES * THREADS * 16;
        static std::atomic<uint64_t> configured{0};
        IT_TRY(allow_dynamic_smem(gat_short_rows_kernel<T, LPR, H>, sbytes, configured));
        const int64_t want = (rows + (THREADS / LPR) - 1) / (THREADS / LPR), most = (int64_t)g->num_sms * IT_GAT_SHORT_BLOCKS;
        const unsigned blocks = (unsigned)(want < most ? want : most);
        IT_LAUNCH(IT_K_GAT_FLAT, bytes, 0, st, gat_short_rows_kernel<T, LPR, H><<<blocks, THREADS, sbytes, st>>>(p, q, pol));
      }
    } else {   // one warp per row: every such list in one launch (they are neighbours), pieces first
      if (chunked) continue;
      chunked = true;
      double all = bytes;
      int b0 = b;
      while (b0 > 0 && g->list_bounds[b0 - 1] > (LPR <= 16 ? IT_SHORT_BELOW : 0)) {
        --b0;
        all += bytes_of(b0, g->h_list_offsets[b0 + 1] - g->h_list_offsets[b0]);
      }
      p.row_lo = g->h_list_offsets[b0];
      static std::atomic<uint64_t> configured{0};
      IT_TRY(allow_dynamic_smem(gat_rows_chunk_kernel<T, LPR, H>, smem, configured));
      p.counter = a.counters + b;
      const unsigned blocks = chunk_grid(p, b == g->n_lists - 1 ? rows : 0, (int64_t)g->num_sms * IT_GAT_CHUNK_BLOCKS);
      IT_LAUNCH(IT_K_GAT_FLAT, all, 0, st, gat_rows_chunk_kernel<T, LPR, H><<<blocks, THREADS, smem, st>>>(p, q, pol));
      p.counter = nullptr;
    }
  }
  IT_CUDA_TRY(cudaGetLastError());
  return IT_OK;
}

}  // namespace
