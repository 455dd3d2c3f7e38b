// fp32 GEMM for CERB_F32 models: out[M][N] = X[M][K] . W[N][K]^T with plain FMA arithmetic
// (tensor cores would round the operands to tf32, which the fp32 contract does not allow).
#include "cerb_internal.cuh"

namespace cerb {

constexpr int TM = 64, TN = 64, TK = 16;
constexpr int kFewTiles = 296;          // 64 x 64 tiles below which the small kernel runs

__global__ void __launch_bounds__(256) gemm_f32_kernel(const float* X, const float* __restrict__ W,
                                                       float* __restrict__ out, int M, int N, int K) {
  __shared__ float sx[TK][TM + 4];
  __shared__ float sw[TK][TN + 4];
  griddep_wait();
  griddep_launch();
  int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  int tx = threadIdx.x % 16, ty = threadIdx.x / 16;     // tx -> n, ty -> m
  float acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += TK) {
    for (int i = threadIdx.x; i < TM * TK; i += 256) {
      int r = i / TK, kk = i % TK;
      int m = m0 + r, k = k0 + kk;
      sx[kk][r] = (m < M && k < K) ? X[(size_t)m * K + k] : 0.f;
      int nn = n0 + r;
      sw[kk][r] = (nn < N && k < K) ? W[(size_t)nn * K + k] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) { a[i] = sx[kk][ty * 4 + i]; b[i] = sw[kk][tx * 4 + i]; }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  for (int i = 0; i < 4; ++i) {
    int m = m0 + ty * 4 + i;
    if (m >= M) continue;
    for (int j = 0; j < 4; ++j) {
      int nn = n0 + tx * 4 + j;
      if (nn < N) out[(size_t)m * N + nn] = acc[i][j];
    }
  }
}

// The same for few output tiles (the small models this path is for: 16 rows x 768 columns x 256).  Such a GEMM is pure
// latency: with the kernel above it was 12 CTAs going through 16 load - wait - multiply rounds one after the other, 16 us for
// 6 MFLOP (a request to the tiny fp32 model: 11.1 ms, 2.8 with this kernel and the attention in fours).  Here a CTA takes
// 16 x 16 outputs, fetches 256 k of both operands in one round, the next 256 while it multiplies, and its eight warps take 32 k
// each; their sums meet in shared memory at the end.
// VEC: the rows of both operands start on 16-byte boundaries (K a multiple of 4, aligned pointers) and come in 16-byte loads;
// otherwise value by value.
// A forward's launches cost what their starts and ends cost, so what stands before and behind its products runs in here (KIND as in
// GemmEpilogue, 0 the product itself): the RMSNorm in front where a row fits one round (NORM: a row is in the registers of 16 threads on
// its way to shared memory), SwiGLU, RoPE and cache append, the residual add behind.  For KIND 1 and 2 a CTA's 16 weight rows are 8 and
// the 8 that belong to them, so that the members of a pair sit 8 lanes apart.  Five launches per layer instead of nine: a 16-node
// verification of four layers of 256 columns 125 -> 90 us, a request of 12 steps 2445 -> 2075; 320 rows 378 -> 353.
// What such a launch needs beside its sum comes behind the rounds, and the kernel behind it is let go there: held through them it took
// the third CTA of an SM, and the next launch's CTAs, with their own fetches, the places and the bandwidth of this one's (four layers of
// 2048 columns, one row: 488 us with separate kernels, 585 so, 475 now; 768 columns, 128 rows 571, 615, 556; 1024 columns, 64 rows 567,
// 499, 506).  (KIND 2 with the norm has 80 registers by itself; held to them it spills.)
constexpr int SM_T = 16, SM_K = 256, SM_LD = SM_K + 4;
struct F32Fused {
  float* act;               // KIND 1: [M][N / 2]
  RopeEpilogue re;          // KIND 2; head_dim 2 * half
  int half;
  const float* gain;        // NORM
  float eps;
};
template <bool VEC, int KIND, bool NORM>
__global__ void __launch_bounds__(256, KIND == 2 && NORM ? 0 : 3) gemm_f32_small_kernel(const float* X, const float* __restrict__ W,
                                                                                         float* out, int M, int N, int K, const F32Fused f) {
  constexpr bool PAIRS = KIND == 1 || KIND == 2;
  __shared__ __align__(16) float sx[SM_T][SM_LD], sw[SM_T][SM_LD];
  __shared__ float red[8][SM_T * SM_T];
  const int m0 = blockIdx.y * SM_T, n0 = blockIdx.x * SM_T;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r = threadIdx.x >> 4, c4 = (threadIdx.x & 15) * 4;     // this thread's pieces: row r, columns c4 + 64 i
  float4 px[4], pw[4];
  auto piece = [&](const float* P, int rows, int row, int k) {
    if (row >= rows || k >= K) return make_float4(0.f, 0.f, 0.f, 0.f);
    const float* at = P + (size_t)row * K + k;
    if constexpr (VEC) return *reinterpret_cast<const float4*>(at);
    return make_float4(at[0], k + 1 < K ? at[1] : 0.f, k + 2 < K ? at[2] : 0.f, k + 3 < K ? at[3] : 0.f);
  };
  // weight row n of this CTA
  auto weight_row = [&](int n) {
    if constexpr (!PAIRS) return n0 + n;
    const int e = blockIdx.x * 8 + (n & 7);                        // feature, or rotation pair over all heads
    if constexpr (KIND == 1) return e < N / 2 ? e + (n >> 3) * (N / 2) : N;
    return e < N / 2 ? e / f.half * 2 * f.half + e % f.half + (n >> 3) * f.half : N;
  };
  const int w_row = weight_row(r);
  auto fetch_w = [&](int k0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) pw[i] = piece(W, N, w_row, k0 + c4 + 64 * i);
  };
  auto fetch_x = [&](int k0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) px[i] = piece(X, M, m0 + r, k0 + c4 + 64 * i);
  };
  fetch_w(0);                                                      // (weights: before the wait)
  float4 pg[NORM ? 4 : 1];
  if constexpr (NORM) {
#pragma unroll
    for (int i = 0; i < 4; ++i) pg[i] = c4 + 64 * i < K ? *reinterpret_cast<const float4*>(f.gain + c4 + 64 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  griddep_wait();
  if constexpr (KIND == 0) griddep_launch();
  fetch_x(0);
  // this thread's output, and what it needs beside the sum
  const int m = m0 + (threadIdx.x >> 4), n = n0 + (threadIdx.x & 15);
  float old = 0.f;
  int kv = -1;
  float2 cs = make_float2(1.f, 0.f);
  auto fetch_rest = [&]() {
    if (KIND == 3 && m < M && n < N) old = out[(size_t)m * N + n];
    if constexpr (KIND == 2) {
      const int e = blockIdx.x * 8 + (threadIdx.x & 7);
      if (m < M && e < N / 2) {
        int b, v;
        locate_row(m, f.re.row_off, f.re.B, f.re.n, b, v);
        const int at = f.re.len[b] + f.re.depth[v], slot = f.re.len[b] + v;
        if (v < f.re.n_active[b] && at < f.re.max_pos && slot < f.re.max_pos) {
          kv = f.re.page_table[(size_t)b * f.re.max_pages + slot / CERB_PAGE] * f.re.H * CERB_PAGE + slot % CERB_PAGE;
          cs = f.re.rope[(size_t)at * f.half + e % f.half];
        }
      }
    }
  };
  if constexpr (NORM) {
    fetch_rest();
    // (K is at most one round: 16 threads hold a row)
    float ss = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) ss += px[i].x * px[i].x + px[i].y * px[i].y + px[i].z * px[i].z + px[i].w * px[i].w;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const float rms = 1.0f / sqrtf(ss / (float)K + f.eps);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      px[i].x = px[i].x * rms * pg[i].x;
      px[i].y = px[i].y * rms * pg[i].y;
      px[i].z = px[i].z * rms * pg[i].z;
      px[i].w = px[i].w * rms * pg[i].w;
    }
  }
  // a lane's outputs: rows tm .. tm + 1, columns tn + 4 j
  const int tm = (lane >> 2) * 2, tn = lane & 3;
  float acc[2][4] = {};
  for (int k0 = 0; k0 < K; k0 += SM_K) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      *reinterpret_cast<float4*>(&sx[r][c4 + 64 * i]) = px[i];
      *reinterpret_cast<float4*>(&sw[r][c4 + 64 * i]) = pw[i];
    }
    __syncthreads();
    if (k0 + SM_K < K) {
      fetch_w(k0 + SM_K);
      fetch_x(k0 + SM_K);
    }
#pragma unroll
    for (int kk = 0; kk < 32; kk += 4) {
      const int k = warp * 32 + kk;
      float4 a[2], b[4];
#pragma unroll
      for (int i = 0; i < 2; ++i) a[i] = *reinterpret_cast<const float4*>(&sx[tm + i][k]);
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = *reinterpret_cast<const float4*>(&sw[tn + 4 * j][k]);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]);
          acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
          acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]);
          acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
        }
    }
    __syncthreads();
  }
  if constexpr (!NORM) fetch_rest();
  if constexpr (KIND != 0) griddep_launch();
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) red[warp][(tm + i) * SM_T + tn + 4 * j] = acc[i][j];
  __syncthreads();
  float v = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) v += red[q][threadIdx.x];
  if constexpr (!PAIRS) {
    if (m < M && n < N) out[(size_t)m * N + n] = KIND == 3 ? old + v : v;
  } else {
    const float other = __shfl_xor_sync(0xffffffffu, v, 8);
    const bool second = threadIdx.x & 8;
    if constexpr (KIND == 1) {
      const int e = blockIdx.x * 8 + (threadIdx.x & 7);
      if (!second && m < M && e < N / 2) f.act[(size_t)m * (N / 2) + e] = v / (1.0f + expf(-v)) * other;
    } else if (kv >= 0) {
      const int e = blockIdx.x * 8 + (threadIdx.x & 7), head = e / f.half, el = e % f.half;
      const int which = head / f.re.H, h = head - which * f.re.H, Dh = 2 * f.half;
      const float o = which == 2 ? v : second ? v * cs.x + other * cs.y : v * cs.x - other * cs.y;
      float* at = which == 0 ? reinterpret_cast<float*>(f.re.q) + ((size_t)m * f.re.H + h) * Dh
                             : reinterpret_cast<float*>(which == 1 ? f.re.kpool : f.re.vpool) + ((size_t)kv + (size_t)h * CERB_PAGE) * Dh;
      at[el + (second ? f.half : 0)] = o;
    }
  }
}

bool gemm_f32_small(int M, int N) { return (long long)((N + TN - 1) / TN) * ((M + TM - 1) / TM) < kFewTiles; }

int launch_gemm_f32_fused(cerb_ctx* c, const float* X, const float* W, int M, int N, int K, const GemmEpilogue& epi, const GemmNorm* norm,
                          cudaStream_t st) {
  if (!gemm_f32_small(M, N) || K % 4 || (((uintptr_t)X | (uintptr_t)W) & 15) || (norm && (K > SM_K || ((uintptr_t)norm->gain & 15)))) return CERB_E_SHAPE;
  F32Fused f = {};
  f.act = (float*)epi.act;
  f.half = c->cfg.head_dim / 2;
  if (epi.kind == 2) f.re = *epi.rope;
  if (norm) { X = norm->x; f.gain = (const float*)norm->gain; f.eps = norm->eps; }
  const int outs = epi.kind == 3 ? SM_T : SM_T / 2, cols = epi.kind == 3 ? N : N / 2;
  const dim3 grid((cols + outs - 1) / outs, (M + SM_T - 1) / SM_T);
  auto go = [&](auto kern) { launch_pdl(kern, grid, dim3(256), 0, st, X, W, epi.x, M, N, K, f); };
  if (epi.kind == 1) norm ? go(gemm_f32_small_kernel<true, 1, true>) : go(gemm_f32_small_kernel<true, 1, false>);
  else if (epi.kind == 2) norm ? go(gemm_f32_small_kernel<true, 2, true>) : go(gemm_f32_small_kernel<true, 2, false>);
  else if (epi.kind == 3 && !norm) go(gemm_f32_small_kernel<true, 3, false>);
  else return CERB_E_ARG;
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

int launch_gemm_f32(cerb_ctx* c, const float* X, const float* W, float* out, int M, int N, int K, cudaStream_t st) {
  // Too few 64 x 64 tiles to fill the GPU: the small ones (us, large / small: 16 x 768 x 256 26 / 14, 512 x 1024 x 256 28 / 21,
  // 1024 x 1024 x 256 with 256 tiles 38 / 39).
  if (gemm_f32_small(M, N)) {
    dim3 small((N + SM_T - 1) / SM_T, (M + SM_T - 1) / SM_T);
    // (a caller without a model may hand over as weights what the kernel in front is still writing)
    const bool vec = K % 4 == 0 && (((uintptr_t)X | (uintptr_t)W) & 15) == 0;
    auto kern = vec ? gemm_f32_small_kernel<true, 0, false> : gemm_f32_small_kernel<false, 0, false>;
    const F32Fused none = {};
    if (c) launch_pdl(kern, small, dim3(256), 0, st, X, W, out, M, N, K, none);
    else kern<<<small, 256, 0, st>>>(X, W, out, M, N, K, none);
    CERB_LAUNCH_CHECK(c);
    return CERB_OK;
  }
  dim3 grid((N + TN - 1) / TN, (M + TM - 1) / TM);
  launch_pdl(gemm_f32_kernel, grid, dim3(256), 0, st, X, W, out, M, N, K);
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

}  // namespace cerb
