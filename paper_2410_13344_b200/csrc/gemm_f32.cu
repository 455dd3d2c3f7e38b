// fp32 GEMM for CERB_F32 models: out[M][N] = X[M][K] . W[N][K]^T with plain FMA arithmetic
// (tensor cores would round the operands to tf32, which the fp32 contract does not allow).
#include "cerb_internal.cuh"

namespace cerb {

constexpr int TM = 64, TN = 64, TK = 16;
constexpr int kFewTiles = 296;          // 64 x 64 tiles below which the small kernel runs

__global__ void __launch_bounds__(256) gemm_f32_kernel(const float* __restrict__ X, const float* __restrict__ W,
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
constexpr int SM_T = 16, SM_K = 256, SM_LD = SM_K + 4;
template <bool VEC>
__global__ void __launch_bounds__(256) gemm_f32_small_kernel(const float* __restrict__ X, const float* __restrict__ W,
                                                             float* __restrict__ out, int M, int N, int K) {
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
  auto fetch_w = [&](int k0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) pw[i] = piece(W, N, n0 + r, k0 + c4 + 64 * i);
  };
  auto fetch_x = [&](int k0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) px[i] = piece(X, M, m0 + r, k0 + c4 + 64 * i);
  };
  fetch_w(0);                                                      // (weights: before the wait)
  griddep_wait();
  griddep_launch();
  fetch_x(0);
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
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) red[warp][(tm + i) * SM_T + tn + 4 * j] = acc[i][j];
  __syncthreads();
  const int m = m0 + (threadIdx.x >> 4), n = n0 + (threadIdx.x & 15);
  float v = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) v += red[q][threadIdx.x];
  if (m < M && n < N) out[(size_t)m * N + n] = v;
}

int launch_gemm_f32(cerb_ctx* c, const float* X, const float* W, float* out, int M, int N, int K, cudaStream_t st) {
  // Too few 64 x 64 tiles to fill the GPU: the small ones (us, large / small: 16 x 768 x 256 26 / 14, 512 x 1024 x 256 28 / 21,
  // 1024 x 1024 x 256 with 256 tiles 38 / 39).
  if ((long long)((N + TN - 1) / TN) * ((M + TM - 1) / TM) < kFewTiles) {
    dim3 small((N + SM_T - 1) / SM_T, (M + SM_T - 1) / SM_T);
    // (a caller without a model may hand over as weights what the kernel in front is still writing)
    const bool vec = K % 4 == 0 && (((uintptr_t)X | (uintptr_t)W) & 15) == 0;
    auto kern = vec ? gemm_f32_small_kernel<true> : gemm_f32_small_kernel<false>;
    if (c) launch_pdl(kern, small, dim3(256), 0, st, X, W, out, M, N, K);
    else kern<<<small, 256, 0, st>>>(X, W, out, M, N, K);
    CERB_LAUNCH_CHECK(c);
    return CERB_OK;
  }
  dim3 grid((N + TN - 1) / TN, (M + TM - 1) / TM);
  launch_pdl(gemm_f32_kernel, grid, dim3(256), 0, st, X, W, out, M, N, K);
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

}  // namespace cerb
