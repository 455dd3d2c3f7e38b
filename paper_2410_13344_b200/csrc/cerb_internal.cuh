// Internal declarations shared by the translation units of libcerb.so.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <vector>

#include "cerb.h"

#define CERB_CUDA_OK(expr)                         \
  do {                                             \
    cudaError_t e__ = (expr);                      \
    if (e__ != cudaSuccess) return CERB_E_CUDA;    \
  } while (0)

#define CERB_TRY(expr)                 \
  do {                                 \
    int rc__ = (expr);                 \
    if (rc__ != CERB_OK) return rc__;  \
  } while (0)

#define CERB_LAUNCH_CHECK(c)                                   \
  do {                                                         \
    if (c) (c)->launches++;                                    \
    if (cudaGetLastError() != cudaSuccess) return CERB_E_CUDA; \
  } while (0)

namespace cerb {

typedef __nv_bfloat16 bf16;

// Programmatic dependent launch: a kernel launched through launch_pdl may begin while its
// predecessor in the stream is still running; it must execute griddep_wait() before it touches
// anything the predecessor writes (or anything the predecessor may still be reading and this
// kernel overwrites).  griddep_launch() lets the next kernel in the stream be scheduled early.
// What another kernel of the stream writes while this one waits is not const __restrict__ here: the compiler may fetch such data through
// the read-only path, which the wait does not order.  (Products of a small fp32 model, compiled for three CTAs to an SM, read the
// residual stream of a layer before.)  Constants (weights, gains, trees, rotations) and what is at least two kernels old may be.
#ifdef __CUDACC__
// Which sequence and which node a row of the step's activation buffers belongs to: with ragged rows (sequences that
// verify a one-node tree next to sequences that verify the whole tree) sequence b starts at row_off[b], otherwise at
// b * n.
__device__ __forceinline__ void locate_row(int row, const int32_t* row_off, int B, int n, int& b, int& v) {
  if (!row_off) { b = row / n; v = row - b * n; return; }
  b = 0;
  while (b + 1 < B && row_off[b + 1] <= row) ++b;
  v = row - row_off[b];
}
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Warp MMA, 16 x 8 x 16, bf16 operands, fp32 sums.
__device__ __forceinline__ void mma_16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
#endif
bool pdl_enabled();
// Budget of every bounded device-side wait, in SM clock cycles (cerb_set_wait_cycles; about 2 s by default).
long long wait_cycles();

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// Same, for a kernel whose CTAs form clusters of `cluster_x` along x.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                      unsigned cluster_x, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster_x;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

constexpr int kPathMax = CERB_MAX_DEPTH + 1;
// Rows of one prefill forward.  A forward streams all the weights whatever its row count, so short chunks pay for the
// stream again and again: a 2048-token prompt of the 7B shape took 73.7 ms in 128-token chunks (16 weight streams,
// 0.23 of the tensor peak).  The sequences of a batch share the rows.  (Up to 2048 rows a forward, and as many tokens of
// every prompt as fit: eight ragged prompts of up to 437 tokens, 2460 in all, left 412 to a second forward, 41.7 ms; 39.3 in one.)
constexpr int kPrefillRows = 4096;
constexpr int kPrefillQuantum = 128;    // tokens per sequence and forward come in multiples of this (the attention window)
constexpr int kGemmRowsPerPass = 256;   // activation rows one tcgen05 pass covers at most (the MMA's N extent; CTA pairs)
constexpr int kGemmMaxSplit = 16;

// Device-side copy of a tree, living in the workspace.
struct TreeDev {
  int32_t* parent;   // [CERB_MAX_NODES]
  int32_t* depth;
  int32_t* head_of;
  int32_t* rank_of;
  uint64_t* anc;     // [CERB_MAX_NODES][CERB_ANC_WORDS]
};
constexpr size_t kTreeSlotBytes = 4 * CERB_MAX_NODES * sizeof(int32_t) + CERB_MAX_NODES * CERB_ANC_WORDS * sizeof(uint64_t);

// Tensor maps for one activation buffer used as the MMA's B operand, one per number of rows fetched at a time.
struct ActMaps {
  CUtensorMap m[8];                     // boxes of 16, 32, ... 128 rows
  const CUtensorMap& box(int rows) const { return m[rows / 16 - 1]; }
};

// Chains of tensor-core accumulations that a product's sums are made of, in blocks of 64 k.  The tensor cores cut a running sum off towards zero at every
// step, so the error of a sum grows with the length of its chains: over all sums like the root of `cubes` per block.
struct Chains {
  int longest = 0;
  double cubes = 0, blocks = 0;
  // a run of n blocks dealt to `chains` accumulators
  void add(int n, int chains) {
    for (int i = 0; i < chains && i < n; ++i) chain((n - i + chains - 1) / chains);
  }
  void chain(int n) {
    if (n > longest) longest = n;
    cubes += (double)n * n * n;
    blocks += n;
  }
  double mean_square() const { return blocks ? cubes / blocks : 0; }
  // (one per cent of the mean square: blocks are whole)
  bool no_longer_than(const Chains& o) const { return longest <= o.longest && mean_square() <= 1.01 * o.mean_square(); }
};

// gemm_rows.cu: how a matrix is cut into one tile per SM, and for up to 32, 64, 96, 128, 192 and 256 rows what runs it; no tiles, or no chains there = not
// for that kernel
constexpr int kRowsClasses = 6;
inline int rows_class_limit(int i) { return i < 4 ? 32 * (i + 1) : 64 * (i - 1); }
inline int rows_class(int M) { return M <= 8 || M > 256 ? -1 : M <= 128 ? (M - 1) / 32 : (M - 1) / 64 + 2; }
struct RowsRing {
  int stages, issuers, chains;
};
struct RowsPlan {
  int groups, tiles;
  bool heads;               // cut by heads (RoPE)
  int parts;                // plain sums: pieces that k is cut into, each a slot of the output
  RowsRing ring[kRowsClasses];
};

// ... and the plain products: a plan for each of these classes, with the maps of all layers.
struct RowsSums {
  RowsPlan plan[kRowsClasses];
  std::vector<CUtensorMap> map[kRowsClasses];
  // which of them is for M rows, or -1
  int at(int M) const {
    const int i = rows_class(M);
    return i >= 0 && plan[i].tiles ? i : -1;
  }
};

}  // namespace cerb

struct cerb_tree {
  int32_t n;
  int32_t slot;
  int32_t max_depth;
  cerb::TreeDev dev;
  std::vector<int32_t> parent, depth;
};

struct cerb_ctx {
  cerb_config cfg;
  bool bf16;
  size_t esize;                       // bytes per model element
  int Mmax;                           // max rows of one forward (max_batch * max_nodes, or a prefill forward's)
  int max_pos;                        // 16 * max_pages
  int head_w[CERB_MAX_HEADS][CERB_MAX_LEVELS + 1];   // state width entering each level
  int head_wmax;

  // weights (device pointers, host arrays)
  const void *embed, *final_norm, *lm_head;
  bool f32_aligned;                   // fp32: every matrix of the layers starts on a 16-byte boundary (gains always do)
  std::vector<const void*> attn_norm, wqkv, wo, mlp_norm, wgu, wd, head_W, head_b, head_fc;
  char *k_pool, *v_pool;
  size_t pool_layer_bytes;
  const int32_t* page_table;

  // tensor maps (bf16 only)
  std::vector<CUtensorMap> tm_wqkv, tm_wo, tm_wgu, tm_wd;
  std::vector<CUtensorMap> tm_wqkv_rot, tm_wgu_pair;   // the same rows gathered for the epilogues above 128 rows
  std::vector<CUtensorMap> tm_wqkv_rows, tm_wgu_rows;  // ... and for those of gemm_rows.cu, where there is a plan
  cerb::RowsPlan rows_qkv, rows_gu;
  cerb::RowsSums rows_wo, rows_wd, rows_lm;
  CUtensorMap tm_lm_head;
  cerb::ActMaps tm_xn, tm_attn, tm_act, tm_hidden, tm_hlast;
  std::vector<CUtensorMap> tm_kpool, tm_vpool;        // per layer

  // workspace carve-out
  int32_t *d_len, *d_len_old, *d_root, *d_nactive, *d_status, *d_lens_in, *d_mode, *d_naccept;
  int32_t *d_path, *d_outtok, *d_argmax, *d_treetok, *d_topk, *d_kper;
  int32_t* d_rowoff;                  // [CERB_MAX_BATCH + 1] first row of every sequence when the rows of a step are ragged
  int32_t* d_iota;                    // [Mmax] 0, 1, 2, ...: the depths of a prefill chunk
  float* d_S;
  void *d_hlast, *d_x, *d_xn, *d_q, *d_attn, *d_act, *d_hidden;
  float *d_part, *d_logits, *d_hlogits;
  float* d_topk_cv;       // per-chunk top-k candidates of the heads' logits: values [B][Hc][kTopkChunks][MAX_TOPK]
  int32_t* d_topk_ci;     // ... and their token ids
  unsigned int* d_gemm_tickets;   // kGemmTickets counters of the GEMM above 128 rows (zero between launches)
  float* d_gemm_fix;      // partial tiles of the GEMM above 128 rows
  size_t part_floats;
  float* d_hstate[2];
  __nv_bfloat16* d_hterms[2];         // bf16 models: the same states as three bf16 terms, [Hc][head_term_cols][head_wmax]
  float2* d_rope;
  char* d_attn_scratch;
  size_t attn_scratch_bytes;
  char* d_tree_store;
  bool tree_used[CERB_MAX_TREES];
  cerb_tree* chain;                   // stands for the prompt tokens of a prefill chunk
  cerb_tree* single;                  // one-node tree for auto-regressive steps

  // pinned host staging
  int32_t* h_stage;                   // [8 * CERB_MAX_BATCH]

  // host-side state
  int B;
  int h_len[CERB_MAX_BATCH];          // upper bound of the committed length per sequence
  const cerb_tree* verified_tree;     // tree of the last cerb_verify not yet accepted
  int64_t launches;
  int last_rows;                      // rows of the last forward (for accounting)
  int sm_count;

  // optional per-family timing (cerb_profile_*)
  bool prof_on;
  int prof_mode;                      // 1: CUDA-event brackets per family; 2: the GEMM kernels stamp their own span
  unsigned long long* d_gemm_clock;   // [2][kGemmClockSlots]: first CTA past its dependency wait, last CTA done (ns)
  int gemm_clock_used;
  std::vector<cudaEvent_t> prof_ev;   // begin/end pairs
  std::vector<int> prof_kind;         // family of each pair
  size_t prof_used;                   // pairs recorded since the last read
};

namespace cerb {

// Rows of one pass of the single-CTA GEMM: 32, 64 or 128.
inline int row_bucket(int rows) {
  int r = 32;
  while (r < rows && r < 128) r <<= 1;
  return r;
}
constexpr int kGemmTickets = 8192;
constexpr int kGemmClockSlots = 4096;
constexpr int kTopkChunks = 16;     // the vocabulary is cut into this many chunks for the heads' top-k

// launch_order.cu: the forward's launch sequence and what each kernel reads ahead of its dependency wait
enum { LO_SET_ACTIVE = 0, LO_NORM_ATTN, LO_GEMM_QKV, LO_ROPE, LO_ATTN, LO_GEMM_WO, LO_NORM_MLP, LO_GEMM_GU, LO_SWIGLU,
       LO_GEMM_DOWN, LO_NORM_FINAL, LO_GEMM_LM, LO_ARGMAX };
// What runs in GEMM epilogues: SwiGLU in the gate-up GEMM, RoPE + cache append in the QKV GEMM, the residual add in the O
// and down GEMMs.
struct Fusion {
  bool swiglu, rope, residual, norm;
};
int launch_order_variant(Fusion f);
int launch_order_layer(int variant, int* ids_out);            // the layer's launches (at most kLayerLaunches)
constexpr int kLayerLaunches = 9;
int launch_order_violations(int variant);

// ---- launch wrappers implemented across the .cu files (all asynchronous on `st`) ----

// glue.cu
int launch_rope_table(cerb_ctx* c, cudaStream_t st);
int launch_fused_norm(cerb_ctx* c, const float* part, int nsplit, size_t split_stride, const int32_t* tok, int tok_stride,
                      int tok_off, int n, const void* gain, void* out, int rows, cudaStream_t st,
                      const int32_t* row_off = nullptr, bool complete = false);
int launch_rope_append(cerb_ctx* c, int layer, const TreeDev& t, const float* part, int nsplit, size_t split_stride,
                       int B, int n, int rows, cudaStream_t st, const int32_t* row_off = nullptr);
int launch_swiglu(cerb_ctx* c, const float* part, int nsplit, size_t split_stride, void* act, int rows, cudaStream_t st);
int launch_argmax_rows(cerb_ctx* c, const float* part, int nsplit, size_t split_stride, int rows, int V, int32_t* out,
                       float* summed, cudaStream_t st);
int launch_set_nactive(cerb_ctx* c, int mode, int a, int b, cudaStream_t st);
int launch_prefill_commit(cerb_ctx* c, cudaStream_t st);

// gemm_f32.cu / gemm_bf16.cu : out[split][M][N] fp32 partial sums of X[M][K] . W[N][K]^T
int launch_gemm_f32(cerb_ctx* c, const float* X, const float* W, float* out, int M, int N, int K, cudaStream_t st);
int gemm_plan_split(int sm_count, int M, int N, int K);
Chains gemm_bf16_chains(int N, int K);               // of up to 128 rows
// What may follow a bf16 GEMM in its epilogue (gemm_few.cu, up to kFewRows rows; gemm_rows.cu, 9 to 256 rows, kinds 1 and 2; gemm_tile.cu, above 128
// rows).
// kind 1 (SwiGLU): W is [gate rows F][up rows F]; act[row][f] = SiLU(gate) * up (bf16).
// kind 2 (RoPE + cache append): W is the QKV matrix [q rows | k rows | v rows] of a model with head_dim 128; q and k are
// rotated at position len + depth, q is written dense and k, v into the paged pools -- what rope_append_kernel does, with the
// same arithmetic in the same order.
// kind 3: the product is added to the fp32 residual stream.
// From 9 to 128 rows separate kernels add the residual (and do the rest where the matrix is not for gemm_rows.cu): the GEMM leaves partial sums there.
struct RopeEpilogue {
  const int32_t *len, *n_active, *depth, *page_table, *row_off;    // as for rope_append_kernel (row_off may be null)
  const float2* rope;       // rotation table [max_pos][64]
  void *q, *kpool, *vpool;  // bf16: q [rows][H * 128]; this layer's pools
  int max_pages, max_pos, n, H, B;
};
struct GemmEpilogue {
  int kind;                 // 0 none, 1 SwiGLU, 2 RoPE + cache append, 3 residual add
  void* act;                // kind 1: [M][F] bf16
  const RopeEpilogue* rope; // kind 2
  float* x;                 // kind 3: [M][N]
};
// gemm_tile.cu: more than 128 rows
struct TilePlan {
  int hf, chains, fill, fills, mchunks, n_act, num_kb, pairs, S, per, sk_tiles;
  long long tiles;          // checked to fit 31 bits before launch
  size_t fix_floats;        // what the plan needs of the fix-up buffer
};
TilePlan make_tile_plan(int M, int N, int K, bool plain, size_t max_fix = ~(size_t)0);
size_t gemm_fix_floats();   // of any plan
Chains gemm_tile_chains(int M, int N, int K);          // of a product with an epilogue
int launch_gemm_tile(cerb_ctx* c, const CUtensorMap* tmW, const ActMaps* tmX, const TilePlan& g, float* out, float* fix, unsigned int* tickets,
                     int M, int N, int32_t* status, cudaStream_t st, const GemmEpilogue* epi = nullptr,
                     unsigned long long* clock_slot = nullptr);
// gemm_few.cu: few rows
constexpr int kFewRows = 8;
struct GemmNorm {           // the GEMM's X is RMSNorm(x) * gain of the residual stream x [M][K]
  const float* x;
  const void* gain;
  float eps;
};
// gemm_f32.cu: fp32, a forward's GEMMs with what stands before and behind them (few output tiles, operands on 16-byte boundaries; norm: K up to 256)
constexpr int kF32NormMax = 256;
bool gemm_f32_small(int M, int N);
int launch_gemm_f32_fused(cerb_ctx* c, const float* X, const float* W, int M, int N, int K, const GemmEpilogue& epi, const GemmNorm* norm,
                          cudaStream_t st);
int launch_gemm_few(cerb_ctx* c, const void* X, const void* W, float* out, int M, int N, int K, cudaStream_t st, const GemmEpilogue* epi = nullptr,
                    const GemmNorm* norm = nullptr, unsigned long long* clock_slot = nullptr);
bool gemm_few_normalises(int M, int K);
// gemm_rows.cu: 9 to 256 rows, kinds 1 and 2, and plain sums; in chains no longer than those of the kernel that takes the product otherwise
bool gemm_rows_takes(const RowsPlan& g, int M);
RowsPlan plan_rows_swiglu(int F, int K);
RowsPlan plan_rows_rope(int n_heads, int head_dim, int K);
Chains gemm_rows_chains(const RowsPlan& g, int M, int K);
Chains gemm_rows_other_chains(int limit, int N, int K);      // of the kernel that takes up to `limit` rows otherwise
int launch_gemm_rows(cerb_ctx* c, const CUtensorMap* tmW, const ActMaps* tmX, const RowsPlan& g, int M, int N, int K, int32_t* status, cudaStream_t st,
                     const GemmEpilogue* epi, float* out = nullptr, unsigned long long* clock_slot = nullptr);
RowsPlan plan_rows_sums(int M, int N, int K, int max_parts);
int launch_gemm_bf16(cerb_ctx* c, const CUtensorMap* tmW, const ActMaps* tmX, float* out, int M, int N, int K,
                     int nsplit, int32_t* status, cudaStream_t st, unsigned long long* clock_slot = nullptr);
int make_weight_map(CUtensorMap* out, const void* W, int N, int K);
int make_gate_up_map(CUtensorMap* out, const void* W, int F, int K);
int make_rotation_map(CUtensorMap* out, const void* W, int heads, int K);
int make_rows_map(CUtensorMap* out, const void* W, int N, int K, int rows);
int make_gate_up_groups(CUtensorMap* out, const void* W, int F, int K, int groups);
int make_rotation_groups(CUtensorMap* out, const void* W, int heads, int K, int groups);
int make_act_map(ActMaps* out, const void* X, int rows_alloc, int K, int box_rows);
int make_act_maps(ActMaps* out, const void* X, int rows_alloc, int K);
int gemm_scratch_slots(int M, int N, int K);
int init_driver_api();

// attention.cu
size_t attn_scratch_bytes(int B, int n, int H, int Dh);
int make_pool_map(CUtensorMap* out, const void* pool, int n_pool_pages, int H, int Dh);
// row_off: first row of every sequence in q / out when the rows of a batch are ragged (device, [B]); null = b * n
// chain: the n nodes of every sequence are consecutive prompt tokens (n may then exceed CERB_MAX_NODES; anc describes a
// chain of 128)
int launch_tree_attention(cerb_ctx* c, const cerb_attn_args* a, const CUtensorMap* tmK, const CUtensorMap* tmV,
                          int sm_count, int32_t* status, cudaStream_t st, const int32_t* row_off = nullptr, bool chain = false);

// heads.cu
inline int head_term_cols(int max_batch) { return (3 * max_batch + 7) / 8 * 8; }
int launch_heads(cerb_ctx* c, const cerb_tree* tree, int32_t* tree_tok, const int32_t* plant, int32_t* topk_out,
                 float* logits_out, cudaStream_t st);

// gate_accept.cu
// host: pinned staging that receives [mode | len | S], CERB_MAX_BATCH words each, or null; host_n, host_tok: device addresses of pinned copies of n_accept
// and out_tok, or null
int launch_gate(cerb_ctx* c, float T, float* S, int32_t* mode, int32_t* nactive_or_null, int n_par, cudaStream_t st, int32_t* host = nullptr);
int launch_accept(cerb_ctx* c, const cerb_tree* tree, const int32_t* tree_tok, const int32_t* n_active,
                  const int32_t* node_argmax, int32_t* n_accept, int32_t* path, int32_t* out_tok, cudaStream_t st,
                  const int32_t* row_off = nullptr, int32_t* host_n = nullptr, int32_t* host_tok = nullptr);

}  // namespace cerb
