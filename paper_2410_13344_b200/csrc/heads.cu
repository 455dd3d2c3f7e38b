// Cerberus decoding heads (Section 4.1).  Every head is a stack of Resblocks
//     plain:      out = SiLU((W h + b) + h)
//     two-input:  h = Concat(h_i, h_{i-1});  out = SiLU((W h + b) + h)
// followed by one FC layer to the vocabulary.  The sequential link sits inside the heads, so all
// heads advance level by level together: one launch per level covers every head (grid.y = head),
// the two-input block of head i reads head i-1's state as it entered the same level.  A level streams its
// weights once, whatever the batch: bf16 models on the tensor cores (head_mma_kernel), fp32 models with
// plain FMA (head_gemv_kernel); bias, residual and SiLU are fused.
// The FC layer reuses the kernel without an epilogue; a per-head top-k (value descending, lower id
// first among equals; per vocabulary chunk, then over the chunks' candidates) and the tree fill follow.
#include "cerb_internal.cuh"

namespace cerb {

namespace {

constexpr int ROWS_PER_WARP = 4;
constexpr int WARPS = 8;
constexpr int ROWS_PER_BLOCK = ROWS_PER_WARP * WARPS;

struct HeadJob {
  const void* W;        // [rows][w_in]
  const void* bias;     // [rows] or null
  int rows;             // output width
  int w0;               // own input width
  int w1;               // appended width (0 for a plain block)
  int src;              // head whose state is appended, or -1
};

struct LevelParams {
  HeadJob job[CERB_MAX_HEADS];
  const float* state_in;    // [B][Hc][wmax]
  float* out;               // state_out [B][Hc][wmax] or logits [B][Hc][out_stride]
  const bf16* terms_in;     // bf16 models: the same state as three bf16 terms, [Hc][cols][wmax], column B term + b
  bf16* terms_out;
  int cols;
  int Hc, wmax, out_stride, B, b0;
  int epilogue;             // 1: SiLU(acc + bias + input[row]); 0: plain product
};

template <typename T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ldf<bf16>(const bf16* p) { return __bfloat162float(*p); }

// fp32 models.
template <int NB>
__global__ void __launch_bounds__(WARPS * 32) head_gemv_kernel(const LevelParams P) {
  extern __shared__ __align__(16) float su[];         // [NB][w]
  const int head = blockIdx.y;
  const HeadJob J = P.job[head];
  const int w = J.w0 + J.w1;
  const int row_base = blockIdx.x * ROWS_PER_BLOCK;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = row_base + warp * ROWS_PER_WARP;
  constexpr int E = 4, AHEAD = 2;
  const float* Wp = reinterpret_cast<const float*>(J.W);
  // the weights' first pieces and the bias come while the kernel in front ends (a level of 4 heads of 256: 4.06 -> 2.64 us)
  float4 wv[AHEAD][ROWS_PER_WARP];
  auto fetch = [&](float4 (&to)[ROWS_PER_WARP], int k) {
#pragma unroll
    for (int i = 0; i < ROWS_PER_WARP; ++i)
      to[i] = r0 + i < J.rows && k < w ? __ldg(reinterpret_cast<const float4*>(Wp + (size_t)(r0 + i) * w + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
#pragma unroll
  for (int a = 0; a < AHEAD; ++a) fetch(wv[a], (a * 32 + lane) * E);
  const int my_row = r0 + lane;                       // lanes 0 .. ROWS_PER_WARP - 1 finish a row each
  const float bias = P.epilogue && lane < ROWS_PER_WARP && my_row < J.rows ? __ldg(reinterpret_cast<const float*>(J.bias) + my_row) : 0.f;
  griddep_wait();
  griddep_launch();
  if (row_base >= J.rows) return;
  for (int nb = 0; nb < NB; ++nb) {
    int seq = P.b0 + nb;
    const float* own = P.state_in + ((size_t)seq * P.Hc + head) * P.wmax;
    const float* oth = J.src >= 0 ? P.state_in + ((size_t)seq * P.Hc + J.src) * P.wmax : own;
    for (int k = threadIdx.x; k < w; k += blockDim.x)
      su[nb * w + k] = seq < P.B ? (k < J.w0 ? own[k] : oth[k - J.w0]) : 0.f;
  }
  __syncthreads();
  float acc[ROWS_PER_WARP][NB];
#pragma unroll
  for (int i = 0; i < ROWS_PER_WARP; ++i)
#pragma unroll
    for (int nb = 0; nb < NB; ++nb) acc[i][nb] = 0.f;
  for (int k0 = lane * E; k0 < w; k0 += 32 * E * AHEAD) {
#pragma unroll
    for (int a = 0; a < AHEAD; ++a) {
      const int k = k0 + a * 32 * E;
      if (k >= w) break;
#pragma unroll
      for (int nb = 0; nb < NB; ++nb) {
        const float4 x = *reinterpret_cast<const float4*>(su + nb * w + k);
#pragma unroll
        for (int i = 0; i < ROWS_PER_WARP; ++i) {
          acc[i][nb] = fmaf(wv[a][i].x, x.x, acc[i][nb]);
          acc[i][nb] = fmaf(wv[a][i].y, x.y, acc[i][nb]);
          acc[i][nb] = fmaf(wv[a][i].z, x.z, acc[i][nb]);
          acc[i][nb] = fmaf(wv[a][i].w, x.w, acc[i][nb]);
        }
      }
      fetch(wv[a], k + 32 * E * AHEAD);
    }
  }
#pragma unroll
  for (int nb = 0; nb < NB; ++nb) {
    float mine = 0.f;
#pragma unroll
    for (int i = 0; i < ROWS_PER_WARP; ++i) {
      for (int o = 16; o > 0; o >>= 1) acc[i][nb] += __shfl_xor_sync(0xffffffffu, acc[i][nb], o);
      if (lane == i) mine = acc[i][nb];
    }
    const int seq = P.b0 + nb;
    if (lane < ROWS_PER_WARP && my_row < J.rows && seq < P.B) {
      float y = mine;
      if (P.epilogue) {
        y += bias + su[nb * w + my_row];
        y = y / (1.0f + expf(-y));
      }
      P.out[((size_t)seq * P.Hc + head) * P.out_stride + my_row] = y;
    }
  }
}

// v = hi + mid + lo, all 24 bits, a term every `stride`.  Cut off, not rounded: the largest values would round to infinity.  An
// infinity is its own first term (inf - inf would make the others, and with them every product, NaN).
__device__ __forceinline__ void store_terms(bf16* at, size_t stride, float v) {
  const bf16 hi = __float2bfloat16_rz(v);
  const float r = isinf(v) ? 0.f : v - __bfloat162float(hi);
  const bf16 mid = __float2bfloat16_rz(r);
  at[0] = hi;
  at[stride] = mid;
  at[2 * stride] = __float2bfloat16_rn(r - __bfloat162float(mid));
}

// One level (or the FC) of every head of a bf16 model, for the whole batch.  Bound by HBM: the weights once, 2.7 GB per
// draft of the 7B shape.  The fp32 states enter the tensor cores as three bf16 terms each (24 bits; the products are exact
// in fp32), so a batch is 3 B MMA columns (all leading terms, then all middle ones, then all last ones) instead of B passes of
// FMAs: with those, a batch of four took 1.90 ms per draft (0.22 of the copy rate), bound by the FMAs and the shared-memory
// loads that feed them.
// The tensor cores cut a sum off, towards zero, at every step, which FMAs do not: with the leading terms of the whole k in one
// chain the logits of the 7B shape were 0.7e-6 to 3.8e-6 (relative, 2-norm) away from float64, FMAs 1.6e-7.  So each pair of
// MMAs of a column tile with leading terms starts from zero and is added to the sum in fp32: 1.2e-7 to 1.4e-7.  The other
// terms are at most 2^-8 of the first; their sums stay in the tensor cores.
// A CTA takes 16 MT 8 / KG weight rows, 16 MT to a warp; KG warps share a row group, each takes every KG-th 32-wide k block,
// and their sums are added in shared memory.  Weights
// go from global memory straight into the A fragments: a lane loads 16 consecutive bytes of a row, and its eight k values
// stand for the k positions that the fragment layout gives that lane in two MMAs; the states are read in the same order.
// The weights of the first blocks are requested before the wait for the level in front.
constexpr int HM_WARPS = 8;
template <int NT, int MT, int U, int KG, int MB>
__global__ void __launch_bounds__(HM_WARPS * 32, MB) head_mma_kernel(const __grid_constant__ LevelParams P) {
  extern __shared__ float red[];                      // [k group][rows][8 NT columns + 1]
  constexpr int RG = HM_WARPS / KG, ROWS = 16 * MT * RG, LD = 8 * NT + 1;
  constexpr int FT = NT <= 3 ? 1 : 2;                 // column tiles with leading terms: B columns, NT = ceil(3 B / 8)
  const int head = blockIdx.y;
  const HeadJob& J = P.job[head];
  const int row_base = blockIdx.x * ROWS;
  if (row_base >= J.rows) {
    griddep_wait();
    return;
  }
  const int w = J.w0 + J.w1;
  const int warp = (threadIdx.x >> 5) % KG, rg = (threadIdx.x >> 5) / KG, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const bf16* Wr[MT][2];
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int e = 0; e < 2; ++e) Wr[m][e] = reinterpret_cast<const bf16*>(J.W) + (size_t)min(row_base + 16 * (m + MT * rg) + 8 * e + g, J.rows - 1) * w;
  const bf16* own = P.terms_in + ((size_t)head * P.cols + g) * P.wmax;
  const bf16* oth = P.terms_in + ((size_t)(J.src >= 0 ? J.src : head) * P.cols + g) * P.wmax - J.w0;
  constexpr int STEP = 32 * KG;
  auto load_w = [&](uint4 (&r)[U][MT][2], int k) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          r[u][m][e] = make_uint4(0, 0, 0, 0);
          if (k + u * STEP < w)
            asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(r[u][m][e].x), "=r"(r[u][m][e].y), "=r"(r[u][m][e].z), "=r"(r[u][m][e].w) : "l"(Wr[m][e] + k + u * STEP));
        }
  };
  auto load_x = [&](uint4 (&r)[U][NT], int k) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const int kk = k + u * STEP;
        r[u][n] = make_uint4(0, 0, 0, 0);
        if (kk < w && 8 * n + g < 3 * P.B) r[u][n] = *reinterpret_cast<const uint4*>((kk < J.w0 ? own : oth) + (size_t)(8 * n) * P.wmax + kk);
      }
  };
  float acc[MT][NT][4];
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n) acc[m][n][0] = acc[m][n][1] = acc[m][n][2] = acc[m][n][3] = 0.f;
  auto multiply = [&](const uint4 (&a)[U][MT][2], const uint4 (&x)[U][NT]) {
    auto step = [&](float* c, int u, int m, int n) {
      mma_16816(c, a[u][m][0].x, a[u][m][1].x, a[u][m][0].y, a[u][m][1].y, x[u][n].x, x[u][n].y);
      mma_16816(c, a[u][m][0].z, a[u][m][1].z, a[u][m][0].w, a[u][m][1].w, x[u][n].z, x[u][n].w);
    };
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          if (n >= FT) {
            step(acc[m][n], u, m, n);
            continue;
          }
          float c[4] = {0.f, 0.f, 0.f, 0.f};
          step(c, u, m, n);
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[m][n][e] += c[e];
        }
  };
  uint4 w0[U][MT][2], w1[U][MT][2], x0[U][NT], x1[U][NT];
  const int k0 = warp * 32 + t * 8;
  load_w(w0, k0);
  griddep_wait();
  griddep_launch();
  load_x(x0, k0);
  for (int k = k0; k - t * 8 < w; k += 2 * U * STEP) {        // (uniform over the warp)
    load_w(w1, k + U * STEP);
    load_x(x1, k + U * STEP);
    multiply(w0, x0);
    load_w(w0, k + 2 * U * STEP);
    load_x(x0, k + 2 * U * STEP);
    multiply(w1, x1);
  }
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        red[(warp * ROWS + 16 * (m + MT * rg) + 8 * (e >> 1) + g) * LD + 8 * n + 2 * t + (e & 1)] = acc[m][n][e];
  __syncthreads();
  for (int i = threadIdx.x; i < ROWS * P.B; i += HM_WARPS * 32) {
    const int rr = i % ROWS, b = i / ROWS, r = row_base + rr;
    if (r >= J.rows) continue;
    float y = 0.f;
#pragma unroll
    for (int q = 0; q < KG; ++q) {
      const float* c = red + (q * ROWS + rr) * LD + b;
      y += c[0] + c[P.B] + c[2 * P.B];
    }
    if (P.epilogue) {
      const int from = r < J.w0 ? head : J.src, at = r < J.w0 ? r : r - J.w0;
      y += ldf(reinterpret_cast<const bf16*>(J.bias) + r) + P.state_in[((size_t)b * P.Hc + from) * P.wmax + at];
      y = y / (1.0f + expf(-y));
      store_terms(P.terms_out + ((size_t)head * P.cols + b) * P.wmax + r, (size_t)P.B * P.wmax, y);
    }
    P.out[((size_t)b * P.Hc + head) * P.out_stride + r] = y;
  }
}

// The last hidden states as the heads' first states (bf16 models: and as terms).
template <typename T>
__global__ void head_init_kernel(const T* h_last, float* __restrict__ state, int Hc, int wmax, int d, bf16* __restrict__ terms,
                                 int cols) {
  griddep_wait();
  griddep_launch();
  const int b = blockIdx.y, h = blockIdx.z, k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= d) return;
  const float v = ldf(h_last + (size_t)b * d + k);
  state[((size_t)b * Hc + h) * wmax + k] = v;
  if (terms) store_terms(terms + ((size_t)h * cols + b) * wmax + k, (size_t)gridDim.y * wmax, v);
}

__device__ __forceinline__ bool better(float va, int ia, float vb, int ib) { return va > vb || (va == vb && ia < ib); }

// The k best of the entries that a warp's lanes hold (N each, in registers), in (value descending, id ascending) order: in
// every round the lanes' own best meet in two warp-wide reductions, and the lane whose entry has won looks through its others again.  Entries
// without an id (0x7fffffff) never win against others.  emit(round, value, id) is called by every lane.
template <int N, typename Emit>
__device__ __forceinline__ void warp_topk(const float (&v)[N], const int (&id)[N], int k, Emit emit) {
  float pv = INFINITY, mine = -INFINITY;
  int pi = -1, mi = 0x7fffffff;
  bool look = true;
  for (int round = 0; round < k; ++round) {
    if (look) {
      mine = -INFINITY;
      mi = 0x7fffffff;
#pragma unroll
      for (int e = 0; e < N; ++e) {
        const bool after = id[e] != 0x7fffffff && (v[e] < pv || (v[e] == pv && id[e] > pi));
        if (after && better(v[e], id[e], mine, mi)) { mine = v[e]; mi = id[e]; }
      }
    }
    // unsigned in the order of the values (+ 0.f: both zeros are one value)
    const unsigned bits = __float_as_uint(mine + 0.f), key = bits & 0x80000000u ? ~bits : bits | 0x80000000u;
    const unsigned top = __reduce_max_sync(0xffffffffu, key);
    pi = __reduce_min_sync(0xffffffffu, key == top ? mi : 0x7fffffff);
    pv = __uint_as_float(top & 0x80000000u ? top & 0x7fffffffu : ~top);
    look = pi == mi;
    emit(round, pv, pi);
  }
}

// Per-head top-k in two steps, bound by their chains of loads and rounds and not by the 0.5 MB they read.  Step 1: the
// vocabulary is cut into kTopkChunks chunks, one CTA per (chunk, head, sequence); each warp finds the k best of its eighth of
// the chunk, 512 entries at a time against the k best so far, and the first warp the k best of the eight lists.  Step 2: one
// warp per (head, sequence) does the same with the chunks' candidates, among which the global k best are, and one CTA per
// sequence then fills the tree.  4 heads x 32000 entries, k = 10: 10.6 and 11.8 us with cold caches; with block-wide rounds
// and the tree filled by a launch of its own 13, 8 and 3 us (a draft of the 7B shape, batch 4: 536 -> 531 us).
constexpr int TK_WARPS = 8, TK_HELD = 16;
__global__ void __launch_bounds__(TK_WARPS * 32) topk_part_kernel(const float* logits, int V, int Hc,
                                                                  const int32_t* __restrict__ kper, float* __restrict__ cand_v,
                                                                  int32_t* __restrict__ cand_i) {
  __shared__ float lv[TK_WARPS][CERB_MAX_TOPK];
  __shared__ int li[TK_WARPS][CERB_MAX_TOPK];
  const int ch = blockIdx.x, h = blockIdx.y, b = blockIdx.z, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* r = logits + ((size_t)b * Hc + h) * V;
  const int k = kper[h];
  griddep_wait();
  griddep_launch();
  const int per = (V + kTopkChunks - 1) / kTopkChunks;
  // (what one warp holds at once goes to one warp: its list is the chunk's)
  const bool one = per <= 32 * TK_HELD;
  const int c1 = min(V, (ch + 1) * per), part = one ? per : (per + TK_WARPS - 1) / TK_WARPS;
  const int j0 = min(c1, ch * per + warp * part), j1 = min(c1, j0 + part);
  if (lane < CERB_MAX_TOPK) { lv[warp][lane] = -INFINITY; li[warp][lane] = 0x7fffffff; }
  for (int base = j0; base < j1; base += 32 * TK_HELD) {
    float v[TK_HELD + 1];
    int id[TK_HELD + 1];
#pragma unroll
    for (int e = 0; e < TK_HELD; ++e) {
      const int j = base + e * 32 + lane;
      v[e] = j < j1 ? r[j] : -INFINITY;
      id[e] = j < j1 ? j : 0x7fffffff;
    }
    __syncwarp();
    v[TK_HELD] = lane < CERB_MAX_TOPK ? lv[warp][lane] : -INFINITY;       // the best so far
    id[TK_HELD] = lane < CERB_MAX_TOPK ? li[warp][lane] : 0x7fffffff;
    __syncwarp();
    warp_topk(v, id, k, [&](int round, float bv, int bi) {
      if (lane == 0) { lv[warp][round] = bv; li[warp][round] = bi; }
    });
  }
  const size_t o = (((size_t)b * Hc + h) * kTopkChunks + ch) * CERB_MAX_TOPK;
  if (one) {
    __syncwarp();
    if (warp == 0 && lane < k) {
      cand_v[o + lane] = lv[0][lane];
      cand_i[o + lane] = li[0][lane] == 0x7fffffff ? -1 : li[0][lane];
    }
    return;
  }
  __syncthreads();
  if (warp == 0) {
    constexpr int N = TK_WARPS * CERB_MAX_TOPK / 32;
    float v[N];
    int id[N];
#pragma unroll
    for (int e = 0; e < N; ++e) {
      v[e] = (&lv[0][0])[e * 32 + lane];
      id[e] = (&li[0][0])[e * 32 + lane];
    }
    warp_topk(v, id, k, [&](int round, float bv, int bi) {
      if (lane == 0) {
        cand_v[o + round] = bv;
        cand_i[o + round] = bi == 0x7fffffff ? -1 : bi;
      }
    });
  }
}

// One CTA per sequence, one warp per head: the merge, then the tree's tokens.
__global__ void __launch_bounds__(CERB_MAX_HEADS * 32) topk_merge_kernel(const float* cand_v, const int32_t* cand_i,
                                                                         int Hc, const int32_t* __restrict__ kper, int32_t* __restrict__ topk,
                                                                         int32_t* __restrict__ topk_copy, const int32_t* __restrict__ root,
                                                                         const int32_t* __restrict__ head_of, const int32_t* __restrict__ rank_of,
                                                                         const int32_t* __restrict__ plant, int n, int32_t* __restrict__ tree_tok) {
  __shared__ int best_s[CERB_MAX_HEADS][CERB_MAX_TOPK];
  const int b = blockIdx.x, h = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // (what the tree is filled from beside the candidates is older than the heads' launches)
  static_assert(CERB_MAX_HEADS * 32 >= CERB_MAX_NODES, "a thread per node");
  const int v_node = threadIdx.x;
  int from_head = 0, from_rank = 0, planted = -1, root_tok = 0;
  if (tree_tok && v_node < n) {
    if (v_node == 0) root_tok = root[b];
    else { from_head = head_of[v_node]; from_rank = rank_of[v_node]; }
    if (plant) planted = plant[(size_t)b * n + v_node];
  }
  const int k = h < Hc ? kper[h] : 0;
  griddep_wait();
  griddep_launch();
  if (h < Hc) {
    const size_t base = ((size_t)b * Hc + h) * kTopkChunks * CERB_MAX_TOPK;
    constexpr int N = kTopkChunks * CERB_MAX_TOPK / 32;
    float v[N];
    int id[N];
#pragma unroll
    for (int e = 0; e < N; ++e) {
      // candidate (chunk, round) = (t / MAX_TOPK, t % MAX_TOPK)
      const int t = e * 32 + lane;
      const bool in = (t % CERB_MAX_TOPK) < k;
      const int c = in ? cand_i[base + t] : -1;
      const float val = in ? cand_v[base + t] : 0.f;
      v[e] = c >= 0 ? val : -INFINITY;
      id[e] = c >= 0 ? c : 0x7fffffff;
    }
    if (lane < CERB_MAX_TOPK) best_s[h][lane] = -1;
    __syncwarp();
    warp_topk(v, id, k, [&](int round, float, int bi) {
      if (lane == 0) best_s[h][round] = bi == 0x7fffffff ? -1 : bi;
    });
    __syncwarp();
    if (lane < CERB_MAX_TOPK) {
      const size_t o = ((size_t)b * Hc + h) * CERB_MAX_TOPK + lane;
      topk[o] = best_s[h][lane];
      if (topk_copy) topk_copy[o] = best_s[h][lane];
    }
  }
  __syncthreads();
  if (!tree_tok || v_node >= n) return;
  tree_tok[(size_t)b * n + v_node] = v_node == 0 ? root_tok : planted >= 0 ? planted : best_s[from_head][from_rank];
}

template <int NT, int MT, int U, int KG, int MB>
int launch_mma(cerb_ctx* c, const LevelParams& P, int max_rows, cudaStream_t st) {
  constexpr int ROWS = 16 * MT * (HM_WARPS / KG);
  constexpr size_t smem = (size_t)KG * ROWS * (8 * NT + 1) * sizeof(float);
  static std::atomic<bool> configured{false};
  if (!configured) {
    CERB_CUDA_OK(cudaFuncSetAttribute(head_mma_kernel<NT, MT, U, KG, MB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    configured = true;
  }
  if (launch_pdl(head_mma_kernel<NT, MT, U, KG, MB>, dim3((max_rows + ROWS - 1) / ROWS, P.Hc), dim3(HM_WARPS * 32), smem, st, P) != cudaSuccess)
    return CERB_E_CUDA;
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

// bf16 models: the number of MMA column tiles decides (us per draft of the 7B shape, HBM floor 410).  Few columns want
// small CTAs, three to an SM (batch 1: 449 against 492 with 32 rows); more columns want two row tiles to a warp, which share
// its state loads (batch 4: 489 against 520), two warps side by side on the same k blocks, whose state loads meet in L1 (batch
// 8: 519 against 524; batch 9: 687 against 712), and from five tiles on, where the states weigh more than the weights on their
// way from L2, three row tiles (batch 11: 782 against 810 with two and 848 with four, which do not fit the registers; batch
// 16: 846, 976, 1130).
int launch_level_mma(cerb_ctx* c, const LevelParams& P, int max_rows, cudaStream_t st) {
  switch ((3 * P.B + 7) / 8) {
    case 1: return launch_mma<1, 1, 2, 8, 3>(c, P, max_rows, st);
    case 2: return launch_mma<2, 2, 1, 8, 2>(c, P, max_rows, st);
    case 3: return launch_mma<3, 2, 1, 4, 2>(c, P, max_rows, st);
    case 4: return launch_mma<4, 2, 2, 4, 1>(c, P, max_rows, st);
    case 5: return launch_mma<5, 3, 1, 8, 1>(c, P, max_rows, st);
    default: return launch_mma<6, 3, 1, 8, 1>(c, P, max_rows, st);
  }
}

int launch_level(cerb_ctx* c, const LevelParams& P, int max_rows, int max_w, cudaStream_t st) {
  dim3 grid((max_rows + ROWS_PER_BLOCK - 1) / ROWS_PER_BLOCK, P.Hc);
  size_t smem1 = (size_t)max_w * sizeof(float);
  static std::atomic<bool> configured{false};
  if (!configured) {
    CERB_CUDA_OK(cudaFuncSetAttribute(head_gemv_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    CERB_CUDA_OK(cudaFuncSetAttribute(head_gemv_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    configured = true;
  }
  LevelParams Q = P;
  if (P.B == 1) {
    Q.b0 = 0;
    launch_pdl(head_gemv_kernel<1>, grid, dim3(WARPS * 32), smem1, st, Q);
    CERB_LAUNCH_CHECK(c);
  } else {
    if (smem1 * 4 > 200 * 1024) return CERB_E_SHAPE;
    for (int b0 = 0; b0 < P.B; b0 += 4) {
      Q.b0 = b0;
      launch_pdl(head_gemv_kernel<4>, grid, dim3(WARPS * 32), smem1 * 4, st, Q);
      CERB_LAUNCH_CHECK(c);
    }
  }
  return CERB_OK;
}

}  // namespace

int launch_heads(cerb_ctx* c, const cerb_tree* tree, int32_t* tree_tok, const int32_t* plant, int32_t* topk_out,
                 float* logits_out, cudaStream_t st) {
  const cerb_config& g = c->cfg;
  const int Hc = g.n_cheads, L = g.n_levels, d = g.d_model, B = c->B;
  if (Hc <= 0) return CERB_E_STATE;
  if (c->bf16) launch_pdl(head_init_kernel<bf16>, dim3((d + 255) / 256, B, Hc), dim3(256), 0, st, (const bf16*)c->d_hlast, c->d_hstate[0], Hc, c->head_wmax, d, c->d_hterms[0], head_term_cols(g.max_batch));
  else launch_pdl(head_init_kernel<float>, dim3((d + 255) / 256, B, Hc), dim3(256), 0, st, (const float*)c->d_hlast, c->d_hstate[0], Hc, c->head_wmax, d, (bf16*)nullptr, 0);
  CERB_LAUNCH_CHECK(c);
  for (int j = 0; j <= L; ++j) {
    LevelParams P;
    P.state_in = c->d_hstate[j & 1];
    P.Hc = Hc; P.wmax = c->head_wmax; P.B = B; P.b0 = 0;
    P.terms_in = c->d_hterms[j & 1]; P.terms_out = c->d_hterms[(j + 1) & 1]; P.cols = head_term_cols(g.max_batch);
    int max_rows = 0, max_w = 0;
    for (int h = 0; h < Hc; ++h) {
      HeadJob& J = P.job[h];
      if (j < L) {
        int src = g.concat_src[h][j];
        J.W = c->head_W[h * L + j];
        J.bias = c->head_b[h * L + j];
        J.w0 = c->head_w[h][j];
        J.w1 = src >= 0 ? c->head_w[src][j] : 0;
        J.src = src;
        J.rows = J.w0 + J.w1;
      } else {
        J.W = c->head_fc[h];
        J.bias = nullptr;
        J.w0 = c->head_w[h][L];
        J.w1 = 0;
        J.src = -1;
        J.rows = g.vocab;
      }
      if (J.rows > max_rows) max_rows = J.rows;
      if (J.w0 + J.w1 > max_w) max_w = J.w0 + J.w1;
    }
    if (j < L) { P.out = c->d_hstate[(j + 1) & 1]; P.out_stride = c->head_wmax; P.epilogue = 1; }
    else { P.out = logits_out ? logits_out : c->d_hlogits; P.out_stride = g.vocab; P.epilogue = 0; }
    if (c->bf16) CERB_TRY(launch_level_mma(c, P, max_rows, st));
    else CERB_TRY(launch_level(c, P, max_rows, max_w, st));
  }
  const float* lg = logits_out ? logits_out : c->d_hlogits;
  static_assert(kTopkChunks * CERB_MAX_TOPK % 32 == 0, "whole warps of candidates in the merge");
  launch_pdl(topk_part_kernel, dim3(kTopkChunks, Hc, B), dim3(TK_WARPS * 32), 0, st, lg, g.vocab, Hc, (const int32_t*)c->d_kper, c->d_topk_cv, c->d_topk_ci);
  CERB_LAUNCH_CHECK(c);
  launch_pdl(topk_merge_kernel, dim3(B), dim3(CERB_MAX_HEADS * 32), 0, st, (const float*)c->d_topk_cv, (const int32_t*)c->d_topk_ci, Hc,
             (const int32_t*)c->d_kper, c->d_topk, topk_out, (const int32_t*)c->d_root, tree ? (const int32_t*)tree->dev.head_of : (const int32_t*)nullptr,
             tree ? (const int32_t*)tree->dev.rank_of : (const int32_t*)nullptr, plant, tree ? tree->n : 0, tree_tok);
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

}  // namespace cerb
