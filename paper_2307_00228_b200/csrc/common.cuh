// Shared declarations of the layer-pass library (host + device helpers, the graph handle,
// the launch entry points of each kernel file).  sm_100a only.
#pragma once

#include <atomic>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include "inferturbo.h"

#define IT_NUM_SMS_FALLBACK 148
#ifndef IT_SMALL_ROWS
#define IT_SMALL_ROWS (1 << 17)
#endif
#ifndef IT_SMALL_EDGES
#define IT_SMALL_EDGES (1 << 21)
#endif
#ifndef IT_SMALL_DENSE
#define IT_SMALL_DENSE 256
#endif
#ifndef IT_SMALL_DENSE_ROWS
#define IT_SMALL_DENSE_ROWS 2048
#endif
#ifndef IT_SMALL_DENSE_EDGES
#define IT_SMALL_DENSE_EDGES (7 << 17)
#endif

// ----------------------------------------------------------------------------- errors
void it_set_error(const char *fmt, ...);

#define IT_CUDA_TRY(expr)                                                            \
  do {                                                                               \
    cudaError_t _e = (expr);                                                         \
    if (_e != cudaSuccess) {                                                         \
      it_set_error("%s failed: %s (%s:%d)", #expr, cudaGetErrorString(_e), __FILE__, \
                   __LINE__);                                                        \
      cudaGetLastError(); /* reported here, not by a later call */                   \
      return (_e == cudaErrorMemoryAllocation) ? IT_ERR_OOM : IT_ERR_CUDA;           \
    }                                                                                \
  } while (0)

#define IT_TRY(expr)               \
  do {                             \
    it_status _s = (expr);         \
    if (_s != IT_OK) return _s;    \
  } while (0)

#define IT_REQUIRE(cond, code, ...) \
  do {                              \
    if (!(cond)) {                  \
      it_set_error(__VA_ARGS__);    \
      return (code);                \
    }                               \
  } while (0)

// ----------------------------------------------------------------------------- instrumentation
enum it_kernel_id {
  IT_K_VALIDATE = 0, IT_K_SPLIT_SCAN, IT_K_SPLIT_FILL, IT_K_BUCKET_SCAN, IT_K_PREP, IT_K_GATHER_FLAT,
  IT_K_GATHER_EMPTY, IT_K_COMBINE, IT_K_GEMM_FP32, IT_K_GEMM_TC, IT_K_GAT_FLAT, IT_K_GAT_EMPTY,
  IT_K_EDGE_MSG, IT_K_AGG_FINISH, IT_K_GEMM2_TC, IT_K_GATHER_SMALL, IT_K_GAT_SMALL,
  IT_K_COUNT
};
// Wraps one kernel launch: counts it and, while profiling is on, brackets it with events on `st`.
struct it_prof_scope {
  it_prof_scope(int kid, double algo_bytes, double algo_flops, cudaStream_t st);
  ~it_prof_scope();
  int slot_;
  cudaStream_t st_;
};
bool it_profile_is_on();
#define IT_LAUNCH(kid, bytes, flops, st, ...) \
  do {                                        \
    it_prof_scope _scope((kid), (bytes), (flops), (st)); \
    __VA_ARGS__;                              \
  } while (0)

// ----------------------------------------------------------------------------- graph handle
// One row as the gather kernels read it: first edge, edge count, and where the
// aggregate goes (vertex id >= 0 for a whole vertex, ~slot in the partial buffer for a piece of one).
struct __align__(16) it_row_meta {
  int64_t j0;
  int32_t len;
  int32_t dest;
};

struct it_graph {
  int64_t n = 0, e = 0;
  int64_t n_src = 0;   // rows of the table the source ids name (= n unless the graph is one part of a partition)
  const void *indptr = nullptr;
  it_itype indptr_type = IT_I64;
  const int32_t *indices = nullptr;
  const float *edge_weights = nullptr;
  const void *edge_feat = nullptr;   // [e, edge_dim] rows in CSR order (borrowed), set by it_graph_set_edge_features
  int32_t edge_dim = 0;
  it_dtype edge_dtype = IT_F32;
  int device = 0;
  int num_sms = IT_NUM_SMS_FALLBACK;

  // derived by the split (library-owned, device; all carved out of one allocation that is kept for the next split)
  char *slab = nullptr;
  size_t slab_bytes = 0;
  mutable std::atomic<bool> used{false};   // the arrays of the present split have been handed out: to a forward pass or to the caller
  int64_t threshold = 0;
  int64_t n_rows = 0;           // R
  int64_t n_split_owners = 0;   // vertices with more than one shadow row
  int64_t *shadow_indptr = nullptr;  // [R+1]
  int32_t *shadow_owner = nullptr;   // [R]
  int64_t *owner_indptr = nullptr;   // [n+1]
  int32_t n_buckets = 0;
  int64_t bucket_bounds[IT_MAX_BUCKETS] = {0};
  int64_t *bucket_offsets = nullptr;  // device [n_buckets+1]
  int32_t *bucket_rows = nullptr;     // [R]
  int *d_status = nullptr;            // device word: set to 1 by a kernel whose bounded wait gave up

  // what the gather walks: the vertices of at most `long_above` edges by degree bucket, one row each, then the pieces of the
  // longer ones (graph.cu: split).  List b holds entries [h_list_offsets[b], h_list_offsets[b + 1]) of list_meta / list_owner,
  // rows of at most list_bounds[b] edges; the pieces are the last list.
  int32_t n_lists = 0;
  int64_t list_bounds[IT_MAX_BUCKETS + 1] = {0};
  int64_t h_list_offsets[IT_MAX_BUCKETS + 2] = {0};
  int64_t h_list_edges[IT_MAX_BUCKETS + 1] = {0};
  it_row_meta *list_meta = nullptr;   // what a gather needs to know about one row, in one 16-byte load
  int32_t *list_owner = nullptr;      // the vertex each row belongs to
  int64_t n_long = 0;                 // vertices gathered in pieces
  int64_t n_partial_rows = 0;         // their pieces: one partial result each
  int32_t *long_owners = nullptr;     // [n_long] ascending vertex ids
  int32_t *piece_long = nullptr;      // [n_partial_rows]: which of long_owners a piece belongs to
  int64_t *piece_ptr = nullptr;       // [n_long + 1]: the pieces of long_owners[k] are partial rows piece_ptr[k] ..., in edge order
};

// Graphs whose layers are bound by launches and latency, not by bytes: one kernel then walks every list of a layer's rows and
// folds the pieces of long vertices itself.  Measured on both sides of the line (two layers, one kernel against kernels by list):
// fp32 64-64-16, 10k vertices / 100k edges 41 against 238 us, 130k / 2M 192 against 402; fp32 128-128 60k / 2M 167 against 219,
// 130k / 2M 244 against 259; GAT 130k / 2M 141 against 195.
// Graphs of IT_SMALL_DENSE_ROWS vertices and more with more than IT_SMALL_DENSE edges each and more than IT_SMALL_DENSE_EDGES in all keep
// the kernels by list: there are whole rows for the warps, and pieces of 128 edges only add partial rows (fp32 mean 64 / bf16 max 64 /
// fp32 max 512 / fp32 sum 128, one kernel against kernels by list: 3000 vertices, 1M edges 74 / 70 / 266 / 66 against 58 / 47 / 183 / 58
// us; 6000, 2M 124 / 107 / 466 / 117 against 80 / 63 / 316 / 89; on the other sides 8000, 2M 144 / 132 / 508 against 140 / 119 / 642;
// 1000, 1.2M 73 / 70 / 270 / 70 against 83 / 71 / 244 / 73, GAT 60 against 76; 3000, 500k 60 / 66 / 191 against 67 / 66 / 216).
static inline bool it_small_graph(const it_graph *g) {
  const bool dense = g->n >= IT_SMALL_DENSE_ROWS && g->e > IT_SMALL_DENSE * g->n && g->e > IT_SMALL_DENSE_EDGES;
  return g->n <= IT_SMALL_ROWS && g->e <= IT_SMALL_EDGES && !dense;
}

// Words of device memory that the gather of one layer needs: the list counters (zeroed by the launch that uses them), then,
// for small graphs, how many pieces of every long vertex are done.
static inline size_t it_gather_words(const it_graph *g) { return IT_MAX_BUCKETS + 1 + (it_small_graph(g) ? (size_t)g->n_long : 0); }
static inline int *it_done_words(int *words) { return words + IT_MAX_BUCKETS + 1; }

#ifdef __CUDACC__
// A kernel launched with it_launch_pdl may start while the kernel before it in the stream is still running: it calls
// it_wait_prior() before it touches global memory (that kernel, and by the same rule every earlier one, has then finished
// and its writes are visible), and it_allow_next() once all its blocks are resident.
__device__ __forceinline__ void it_wait_prior() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void it_allow_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
cudaError_t it_launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st; cfg.attrs = &attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#endif

static inline size_t it_align_up(size_t x, size_t a = 256) { return (x + a - 1) / a * a; }

// ELU on the device.  The negative branch is exp(x) - 1 with the hardware exponential (absolute error below 1e-6,
// a handful of instructions where expm1f costs a few dozen in the end-of-row code of every short row); close to
// zero, where that difference cancels, the three-term series x + x^2/2 + x^3/6 takes over (relative error below
// 2e-6 at the switch point x = -1/32 and falling towards 0), so the result is relatively accurate everywhere.
#ifdef __CUDACC__
// e^x by the hardware's 2^x; results below 2^-126 are flushed to zero (an attention weight that small against the largest
// one, which is 1, or an e^x of which 1 is subtracted).  Without the flush the compiler guards every exponential with
// three more instructions.
__device__ __forceinline__ float it_exp(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x * 1.4426950408889634f));
  return r;
}
__device__ __forceinline__ float it_elu(float x) {
  const float series = x * fmaf(x, fmaf(x, 1.f / 6.f, 0.5f), 1.f);
  return x > 0.f ? x : (x > -0.03125f ? series : it_exp(x) - 1.f);
}
#endif
static inline int it_dtype_size(it_dtype t) { return t == IT_F32 ? 4 : 2; }

// ----------------------------------------------------------------------------- gather.cu
// What a gather / combine kernel does with the finished aggregate of vertex v.
enum it_epilogue_kind {
  IT_EPI_STORE = 0,      // dst[v, :] = agg                      (feat dtype)
  IT_EPI_ADD_ACT = 1,    // dst[v, :] = act(self[v, :] + agg)    (both feat dtype)
  IT_EPI_BIAS_ACT = 2,   // dst[v, :] = act(bias + agg)          (bias fp32 [dim] or NULL)
  IT_EPI_RAW_F32 = 3     // dst[v, :] = the raw reduce in fp32: plain sum (mean undivided), max or min, and the identity of
                         // the reduce (0, -inf, +inf) for a row without edges: one part's share of a partial-gather
};

struct it_gather_args {
  const it_graph *g;
  it_gather_op op;         // SUM / MEAN / MAX
  int use_edge_weights;
  it_dtype dtype;          // of src rows and of dst rows
  int dim;                 // elements of a row that are gathered (any multiple of 16 bytes)
  const void *src;         // rows that are gathered: row u starts at src + u * src_ld elements
  int src_ld;              // 0 means dim
  int per_edge_rows;       // 1: src is [n_edges, dim] and row j belongs to edge j (edge features); 0: rows are looked up by source vertex
  float *partials;         // [n_partial_rows, dim] fp32 scratch; NULL: long vertices are reduced whole, one block each
  int *counters;           // it_gather_words() device words of scratch (see there)
  int zeroed;              // 1: the second part of them is zero already (and is left so)
  void *dst;               // row v starts at dst + v * dst_ld elements and takes dim of them
  int dst_ld;              // 0 means dim
  it_epilogue_kind epi;
  const void *self_term;   // IT_EPI_ADD_ACT only: row v starts at self_term + v * self_ld elements (stored like the rows)
  int self_ld;             // 0 means dim
  const float *bias;       // [dim] fp32 or NULL, IT_EPI_BIAS_ACT only
  it_act act;              // IT_EPI_ADD_ACT and IT_EPI_BIAS_ACT
};
it_status it_launch_gather(const it_gather_args &a, cudaStream_t stream);

// What the vertices without in-edges (entries [row_lo, row_hi) of the list) end up with.
enum it_empty_kind { IT_EMPTY_VALUE = 0 /* every entry `value` */, IT_EMPTY_BIAS = 1 /* act(bias[i]), NULL: act(0) */, IT_EMPTY_SELF = 2 /* act(self[v, i]) */ };
struct it_empty_rows_args {
  const it_graph *g;
  int64_t row_lo, row_hi;
  it_empty_kind kind;
  void *dst;
  int64_t pitch;           // bytes from one row of dst to the next
  const void *self;        // rows of dtype
  int64_t self_pitch;
  int dim;                 // entries written
  it_dtype dtype;          // of dst
  float value;
  const float *bias;
  it_act act;
};
it_status it_launch_empty_rows(const it_empty_rows_args &a, int kid, double bytes, cudaStream_t stream);

// ----------------------------------------------------------------------------- gat.cu
struct it_gat_args {
  const it_graph *g;
  it_dtype dtype;
  int heads, head_dim;
  const void *z;          // [n, heads*head_dim] messages
  const float *scores;    // [n_src, 2*heads]: source scores of the vertex, then its destination scores
  const float *scores_dst;   // the same layout, row v = local destination v (scores + first_vertex * 2*heads for a part; NULL: scores)
  int per_edge_rows;      // 1: z is [n_edges, dim], row j belonging to edge j
  int per_edge_scores;    // 1: src_scores is [n_edges, heads], row j belonging to edge j (edge features in the logits)
  const float *src_scores;   // [rows, heads], dense: the source-side logit term that is read per edge (row = source vertex, or the
                             // edge itself with per_edge_scores); NULL: the first half of the rows of `scores`
  float *partials;        // it_gat_partial_bytes() of fp32 scratch; NULL: long vertices are reduced whole, one block each
  int *counters;          // it_gather_words() device words of scratch (see there)
  int zeroed;             // 1: the second part of them is zero already (and is left so)
  float slope;
  const float *bias;      // may be NULL
  it_act act;
  void *dst;              // [n, heads*head_dim]
};
it_status it_launch_gat(const it_gat_args &a, cudaStream_t stream);
// Whether the reduce takes this shape with the weights of many edges at a time (then per-edge logit terms need no copies of
// the source rows in edge order).
bool it_gat_batched(it_dtype dtype, int heads, int head_dim);
size_t it_gat_partial_bytes(const it_graph *g, int dim, int heads);

// ----------------------------------------------------------------------------- apply.cu
// C[M, NB] = X1[M, K1] * B[0:K1, :] + X2[M, K2] * B[K1:K1+K2, :]   (X2 may be NULL, K2 = 0)
// B is an fp32 [K1+K2, NB] matrix assembled by it_launch_prep_weights.  Column ranges of C
// go to up to three destinations:
//   [0, n0)        -> out0 (dtype dt0) = act0(C + bias0)
//   [n0, n0+n1)    -> out1 (dtype dt1), raw
//   [n0+n1, NB)    -> out2 (fp32), raw, row stride n2 = NB - n0 - n1
// The rows of such a product as messages of the edges of a graph (bf16 tensor-core path): reduced by destination in its epilogue, or stored.
#define IT_MSG_TILE 128          // edges per tile
enum it_msg_mode { IT_MSG_SUM = 0, IT_MSG_WSUM = 1 /* w: times the edge's weight */, IT_MSG_WMAX = 2, IT_MSG_WMIN = 3, IT_MSG_MAX = 4, IT_MSG_MIN = 5,
                   IT_MSG_STORE = 6 /* not reduced: row m of out0 is edge m's, the fields below are unused */ };
struct it_tc_reduce {
  const void *indptr;            // of the graph
  int indptr64;
  const int32_t *tile_first;     // [tiles] the vertex that edge IT_MSG_TILE * t belongs to
  const int32_t *ends;           // [tiles * IT_MSG_TILE] the vertex whose last edge this is, or -1
  float *partial;                // [tiles][2][dim]: what a vertex that crosses tiles has in a tile where it does not begin / does begin
  const float *weights;          // of the edges, or NULL
  void *dst;                     // bf16 rows: the reduce of every vertex
  int dst_ld, dim;
  it_msg_mode mode;
  int is_mean;
};
struct it_gemm_args {
  int64_t M;
  it_dtype x_dtype;
  const void *X1; int K1;
  const void *X2; int K2;
  const float *B; int NB;
  int n0; void *out0; it_dtype dt0; const float *bias0; it_act act0;
  int n1; void *out1; it_dtype dt1;
  void *out2;
  // tensor-core path, the shapes of it_tc_adds_rows: row m = act0(round(C + bias0) + add_rows[add_idx[m], :]), rows of n0 elements
  // of dt0; `round` to dt0, as if the product had been stored and read back.  Row m is edge m: reduced (out0 unused) or stored
  const void *add_rows; const int32_t *add_idx; it_tc_reduce reduce;
  uint32_t spin_limit;   // tensor-core path: polls after which a barrier wait gives up (0 = the default)
  int no_loads;          // tensor-core path, test hook: issue no operand copies
};
it_status it_launch_gemm(const it_gemm_args &a, cudaStream_t stream);

enum it_prep_kind { IT_PREP_SAGE = 0, IT_PREP_SAGE_REORDER = 1, IT_PREP_GAT = 2, IT_PREP_DENSE = 3 };   // DENSE: B = W [in, out] as it is
// Assemble the fp32 B matrix for a layer (K = its row count): SAGE and dense / GCN: a copy of W [K, out]; REORDER [in, 2*out] =
// [W_self | W_neigh]; GAT [in, out + 2*heads] = [W | W a_src | W a_dst].
it_status it_launch_prep_weights(it_prep_kind kind, const it_layer_desc *layer, int K, float *B,
                                 cudaStream_t stream);

// ----------------------------------------------------------------------------- apply_tc.cu
// The same product on the tensor cores (tcgen05 + TMEM + TMA).  Needs operand rows that are multiples of 16
// bytes (K1, K2 are padded to whole 128-byte k-blocks with zeros) and, for fp32, n0 and n1 multiples of 16 (bf16 outputs of any
// width are padded: the products are exact either way, where fp32 splits its operands); computes the n0 + n1 columns and, for GAT, the
// attention scores [M, 2*heads] in its epilogue (a.B, a.NB and a.out2 are not used).  B is the
// matrix written by it_launch_prep_weights_tc: bf16 [NB, Kp] or fp32 [2, NB, Kp] (hi, lo), K-major, Kp = padded K1 + padded K2.
bool it_tc_supported(const it_gemm_args &a, int heads, int head_dim, bool want_scores);
struct it_prep_tc {
  int kind, in_dim, out_dim, w_is_bf16, NB;   // NB: columns with their padding; columns of no weight are zero
  int seg;                // IT_PREP_SAGE_REORDER: first column of the neighbour half
  int K1, K1p, K2, K2p;   // rows of W behind X1 / X2, and the same rounded up to whole k-blocks (the padding is zero)
  const void *W;
  void *B;   // bf16 [NB, K1p + K2p]  or  fp32 [2, NB, K1p + K2p] (hi, lo)
};
it_prep_tc it_prep_tc_of(it_prep_kind kind, const it_layer_desc *layer, int NB, int seg, int K1, int K2, void *B);
// How the product's columns are laid out: each output padded to a multiple of 16 columns, all of them to whole splits.
// stream: the weights are read again with every row tile instead of staying in shared memory.
struct it_tc_cols { int n0p, n1p, n_splits, nbc, NB, stream; };
bool it_tc_columns(const it_gemm_args &a, int head_dim, bool want_scores, it_tc_cols *out);
size_t it_prep_tc_bytes(const it_prep_tc &p);
// Several weight matrices and `words` zeroed words in as few launches as possible.
it_status it_launch_prep_weights_tc(const it_prep_tc *list, int count, int *zero, size_t words, cudaStream_t stream);
bool it_tc_adds_rows(const it_gemm_args &a);
it_status it_launch_gemm_tc(const it_gemm_args &a, const void *B, const float *att_src, const float *att_dst,
                            int heads, int head_dim, float *scores, int num_sms, int *status, cudaStream_t stream);

// The update of one layer and the transform of the next as one kernel (bf16 only): H = act1([X1 | X2] B1 + bias1) is
// rounded to bf16 and multiplied by B2 without leaving the SM; columns [0, n0) of H B2, plus bias0, go to out0 and
// columns [n0, n0 + n1) to out1.  N1 (columns of H), n0 and n1 must be multiples of 64.
struct it_gemm2_args {
  int64_t M;
  const void *X1; int K1;
  const void *X2; int K2;
  int N1; const float *bias1; it_act act1;
  int n0; void *out0; const float *bias0;
  int n1; void *out1;
  uint32_t spin_limit;   // polls after which a barrier wait gives up (0 = the default)
  int no_loads;          // test hook: issue no operand copies
};
bool it_tc2_supported(const it_gemm2_args &a);
it_status it_launch_gemm2_tc(const it_gemm2_args &a, const void *B1, const void *B2, int num_sms, int *status, cudaStream_t stream);

// ----------------------------------------------------------------------------- message.cu
// Learned messages that their product reduces: which vertex every tile of edges starts in, and where vertices end ...
it_status it_launch_message_tiles(const it_graph *g, int32_t *tile_first, int32_t *ends, cudaStream_t stream);
// ... and, after the product, the vertices that cross tiles and those without edges.
it_status it_launch_message_combine(const it_graph *g, const it_tc_reduce &q, cudaStream_t stream);
// Learned messages, edge by edge: M[j, :] = act(P[indices[j], :] + M[j, :]) in place (M arrives holding the per-edge
// part Q), rows of `dim` elements of `dtype` (a multiple of 16 bytes).
it_status it_launch_edge_messages(const it_graph *g, it_dtype dtype, int dim, const void *P, void *M, it_act act, cudaStream_t stream);
// GAT with edge features: Zj[j, :] = Z[indices[j], :] (unless Zj is NULL) and sc[j, h] = scores[indices[j], h] + att_edge[h, :] . ef[j, :].
it_status it_launch_gat_edge_rows(const it_graph *g, it_dtype dtype, int dim, int heads, const void *Z, const float *scores,
                                  const float *att_edge, void *Zj, float *sc, cudaStream_t stream);
// dense[v, :] = scores[v, 0:heads]: the source scores on their own, 16 bytes per vertex for 4 heads instead of a 32-byte
// row shared with the destination scores (the reduce reads one per edge, at random).
it_status it_launch_compact_scores(int64_t n, int heads, const float *scores, float *dense, cudaStream_t stream);
// out[v, :] = raw[v, :] * scale[v] (0 where scale[v] = 0), fp32 -> dtype.
it_status it_launch_aggregate_finish(int64_t n, int dim, it_dtype dtype, const float *raw, const float *scale, void *out, cudaStream_t stream);
