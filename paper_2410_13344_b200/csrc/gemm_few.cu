// GEMM of few rows: out[M][N] = X[M][K] . W[N][K]^T, bf16 operands, fp32 sums, M up to kFewRows.
//
// Bound by HBM: the weights once.  What a step of one row costs beyond that is the start and the end of every launch, and the
// passes behind it.  So no tensor memory, no descriptors, no ring to set up and no partial sums: a CTA owns 16 weight rows
// over the whole of k, each of its eight warps an eighth of it.  The weights go from global memory straight into the A
// fragments of warp MMAs: a lane loads 16 consecutive bytes of a row, and its eight k values stand for the k positions that
// the fragment layout gives that lane in two MMAs; X is read in the same order.  The warps' sums meet in shared memory.
// Since every output has its one owner, what follows a GEMM runs here (SwiGLU, RoPE and cache append, the residual add), and
// with very few rows the RMSNorm in front does too, in every CTA for itself.
//
// The CTAs are persistent, two to an SM, and their loads run two rounds (64 KB per CTA) ahead, over the end of a tile into the
// next one, and at the start ahead of the wait for the kernel in front.  Loads in flight occupy the L1, so the kernel asks for
// no more shared memory than it needs: with the largest share of it a step took 1.6 times as long.
//
// 7B shape, 16 layers and LM head, 1000 tokens before, us per forward of 1 / 2 / 4 / 8 rows: 1410 / 1381 / 1551 / 1597; with the
// tensor-memory tiles of gemm_bf16.cu, whose partial sums then meet in separate kernels, 1664 / 1623 / 1648 / 1643 (4 and 8 rows
// as one tree).  From nine rows on, a second column tile per MMA row and twice the activation reads cost more than that: 12
// rows 1868 against 1657.
#include <string.h>

#include "cerb_internal.cuh"

namespace cerb {

namespace {

constexpr int WARPS = 8;
constexpr int U = 4;                 // 32-wide k blocks of a round
constexpr int ROWS = 16, LD = kFewRows + 1, ROUND = 32 * U;
constexpr int CTAS = 2 * 148;

struct FewParams {
  const bf16* X;
  const bf16* W;
  float* out;               // KIND 0: [M][N]; KIND 3: the residual stream [M][N]
  bf16* act;                // KIND 1: [M][F]
  RopeEpilogue re;          // KIND 2
  int M, N, K, F;
  int tiles, rounds, range;
  const float* x;           // NORM: X is RMSNorm(x) * gain, x [M][K] fp32
  const bf16* gain;
  float eps;
  unsigned long long* clk;
};

// KIND as in GemmEpilogue.  A tile's 16 rows are neighbours (0, 3), or eight and the eight that belong to them (1: gate, up; 2:
// elements i and i + 64 of a head).
template <int KIND, bool NORM>
__global__ void __launch_bounds__(WARPS * 32, 2) gemm_few_kernel(const __grid_constant__ FewParams p) {
  constexpr bool PAIRS = KIND == 1 || KIND == 2;
  constexpr int OUTS = PAIRS ? ROWS / 2 : ROWS;
  __shared__ float red_s[2][WARPS * ROWS * LD];              // [tile's parity][warp][row][column + 1]
  extern __shared__ __align__(16) bf16 xs[];                 // NORM: the normalised rows, then the gains; [.][K + 32]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int K = p.K;
  // a tile's first row (of a pair: its first member)
  auto first_row = [](int tile) { return KIND == 2 ? (tile / (64 / OUTS)) * 128 + (tile % (64 / OUTS)) * OUTS : tile * OUTS; };
  const bf16* Wr[2];
  const int k0 = warp * p.range + t * 8, k1 = min(K, (warp + 1) * p.range);     // this warp's part of k
  int load_tile = blockIdx.x, load_k = k0;                   // what the next load_w fetches
  auto set_rows = [&]() {
    const int r0 = first_row(load_tile) + g;
    const int r1 = KIND == 1 ? min(r0, p.F - 1) + p.F : KIND == 2 ? r0 + 64 : r0 + 8;
    Wr[0] = p.W + (size_t)min(r0, (KIND == 1 ? p.F : p.N) - 1) * K;
    Wr[1] = p.W + (size_t)min(r1, p.N - 1) * K;
  };
  auto load_w = [&](uint4 (&r)[U][2]) {
    const int end = load_tile < p.tiles ? k1 : 0;
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        r[u][e] = make_uint4(0, 0, 0, 0);
        if (load_k + u * 32 < end)
          asm volatile("ld.global.nc.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(r[u][e].x), "=r"(r[u][e].y), "=r"(r[u][e].z), "=r"(r[u][e].w) : "l"(Wr[e] + load_k + u * 32));
      }
  };
  auto load_x = [&](uint4 (&r)[U], int k) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      r[u] = make_uint4(0, 0, 0, 0);
      if (k + u * 32 < k1 && g < p.M)
        r[u] = *reinterpret_cast<const uint4*>(NORM ? xs + g * (K + 32) + k + u * 32 : p.X + (size_t)g * K + k + u * 32);
    }
  };
  // (two accumulators in turn: the tensor cores cut the sum off at every step, so half the steps is half the error)
  float acc[2][4];
  auto multiply = [&](const uint4 (&a)[U][2], const uint4 (&x)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      mma_16816(acc[0], a[u][0].x, a[u][1].x, a[u][0].y, a[u][1].y, x[u].x, x[u].y);
      mma_16816(acc[1], a[u][0].z, a[u][1].z, a[u][0].w, a[u][1].w, x[u].z, x[u].w);
    }
  };
  uint4 w0[U][2], w1[U][2], x0[U], x1[U];
  set_rows();
  load_w(w0);
  load_k += ROUND;
  load_w(w1);
  if constexpr (NORM)
    for (int j = threadIdx.x * 4; j < K; j += WARPS * 32 * 4)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(xs + p.M * (K + 32) + j)), "l"(p.gain + j) : "memory");
  griddep_wait();
  if (p.clk && threadIdx.x == 0) atomicMin(p.clk, globaltimer_ns());
  griddep_launch();
  if constexpr (NORM) {
    // every CTA normalises the rows for itself, while its first weights are on their way
    __shared__ float ss_s[kFewRows][WARPS];
    for (int m = 0; m < p.M; ++m) {
      const float* xr = p.x + (size_t)m * K;
      float ss = 0.f;
#pragma unroll 4
      for (int j = threadIdx.x * 4; j < K; j += WARPS * 32 * 4) {
        const float4 v = *reinterpret_cast<const float4*>(xr + j);
        ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      if (lane == 0) ss_s[m][warp] = ss;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    for (int m = 0; m < p.M; ++m) {
      float ss = 0.f;
#pragma unroll
      for (int w = 0; w < WARPS; ++w) ss += ss_s[m][w];
      const float r = 1.0f / sqrtf(ss / (float)K + p.eps);
      const float* xr = p.x + (size_t)m * K;
#pragma unroll 4
      for (int j = threadIdx.x * 4; j < K; j += WARPS * 32 * 4) {
        const float4 v = *reinterpret_cast<const float4*>(xr + j);
        const __nv_bfloat162* gp = reinterpret_cast<const __nv_bfloat162*>(xs + p.M * (K + 32) + j);
        const float2 g0 = __bfloat1622float2(gp[0]), g1 = __bfloat1622float2(gp[1]);
        __nv_bfloat162* o = reinterpret_cast<__nv_bfloat162*>(xs + m * (K + 32) + j);
        o[0] = __floats2bfloat162_rn(v.x * r * g0.x, v.y * r * g0.y);
        o[1] = __floats2bfloat162_rn(v.z * r * g1.x, v.w * r * g1.y);
      }
    }
    __syncthreads();
  }
  load_x(x0, k0);
  load_x(x1, k0 + ROUND);
  // thread: row threadIdx.x % OUTS of the tile (of a pair: its first member), activation row threadIdx.x / OUTS
  const int m = threadIdx.x / OUTS, rr = threadIdx.x % OUTS;
  int pos = -1, kv = -1;
  if (KIND == 2 && m < p.M) {
    const RopeEpilogue& e = p.re;
    int b, v;
    locate_row(m, e.row_off, e.B, e.n, b, v);
    const int at = e.len[b] + e.depth[v], slot = e.len[b] + v;
    if (v < e.n_active[b] && at < e.max_pos && slot < e.max_pos) {
      pos = at;
      kv = e.page_table[(size_t)b * e.max_pages + slot / CERB_PAGE] * e.H * CERB_PAGE + slot % CERB_PAGE;
    }
  }
  int parity = 0;
  for (int tile = blockIdx.x; tile < p.tiles; tile += gridDim.x, parity ^= 1) {
    const int first = first_row(tile);
    const float old = KIND == 3 && m < p.M && first + rr < p.N ? p.out[(size_t)m * p.N + first + rr] : 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[0][e] = acc[1][e] = 0.f;
    // rounds in pairs (p.rounds of them); the loads run two rounds ahead, over the end of the tile into the next
    for (int q = 0; q < p.rounds; q += 2) {
      multiply(w0, x0);
      if (q + 2 < p.rounds) {
        load_k = k0 + (q + 2) * ROUND;
      } else {
        load_tile += gridDim.x;
        load_k = k0;
        set_rows();
      }
      load_w(w0);
      load_x(x0, load_k);
      load_k += ROUND;
      multiply(w1, x1);
      load_w(w1);
      load_x(x1, load_k);
    }
    float* red = red_s[parity];
#pragma unroll
    for (int e = 0; e < 4; ++e) red[(warp * ROWS + 8 * (e >> 1) + g) * LD + 2 * t + (e & 1)] = acc[0][e] + acc[1][e];
    __syncthreads();
    if (m >= p.M) continue;
    auto sum = [&](int row) {
      float s = 0.f;
#pragma unroll
      for (int q = 0; q < WARPS; ++q) s += red[(q * ROWS + row) * LD + m];
      return s;
    };
    if constexpr (!PAIRS) {
      if (first + rr < p.N) p.out[(size_t)m * p.N + first + rr] = KIND == 3 ? old + sum(rr) : sum(rr);
    } else {
      float a = sum(rr), b = sum(rr + 8);
      if constexpr (KIND == 1) {
        if (first + rr < p.F) p.act[(size_t)m * p.F + first + rr] = __float2bfloat16_rn(a / (1.0f + expf(-a)) * b);
      } else {
        if (kv < 0) continue;
        const RopeEpilogue& e = p.re;
        const int unit = first >> 7, el = (first & 127) + rr, which = unit / e.H, h = unit - which * e.H;
        if (which < 2) {
          const float2 cs = e.rope[(size_t)pos * 64 + el];
          const float o1 = a * cs.x - b * cs.y;
          b = b * cs.x + a * cs.y;
          a = o1;
        }
        bf16* o = which == 0 ? reinterpret_cast<bf16*>(e.q) + ((size_t)m * e.H + h) * 128 + el
                             : reinterpret_cast<bf16*>(which == 1 ? e.kpool : e.vpool) + ((size_t)kv + (size_t)h * CERB_PAGE) * 128 + el;
        o[0] = __float2bfloat16_rn(a);
        o[64] = __float2bfloat16_rn(b);
      }
    }
  }
  if (p.clk && threadIdx.x == 0) atomicMax(p.clk + kGemmClockSlots, globaltimer_ns());
}

// Rows whose norm a GEMM computes itself: as many as fit 25 KB of shared memory with the gains, two of 4096 columns.  (One
// row: 1419 us for the forward above instead of 1513 with a norm kernel; eight: 2154 instead of 1793, their rows' loads queue
// behind the weights that every CTA has in flight.)
constexpr size_t kNormSmem = 25 * 1024;
size_t norm_smem(int M, int K) { return (size_t)(M + 1) * (K + 32) * sizeof(bf16); }

template <int KIND, bool NORM>
int launch(FewParams p, cudaStream_t st) {
  constexpr int OUTS = KIND == 1 || KIND == 2 ? ROWS / 2 : ROWS;
  p.tiles = ((KIND == 1 ? p.F : KIND == 2 ? p.N / 2 : p.N) + OUTS - 1) / OUTS;
  const int rounds = (p.K + WARPS * ROUND - 1) / (WARPS * ROUND);
  p.range = rounds * ROUND;
  p.rounds = (rounds + 1) & ~1;
  auto kern = gemm_few_kernel<KIND, NORM>;
  static std::atomic<bool> configured{false};
  if (!configured) {
    // the share of the SM's memory that two CTAs need as shared memory; the rest is L1
    constexpr size_t need = 2 * (2 * WARPS * ROWS * LD * sizeof(float) + (NORM ? kNormSmem : 0) + 1024), all = 228 * 1024;
    if (NORM) CERB_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kNormSmem));
    CERB_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)((need * 100 + all - 1) / all)));
    configured = true;
  }
  return launch_pdl(kern, dim3(p.tiles < CTAS ? p.tiles : CTAS), dim3(WARPS * 32), NORM ? norm_smem(p.M, p.K) : 0, st, p) == cudaSuccess
             ? CERB_OK : CERB_E_CUDA;
}

}  // namespace

bool gemm_few_normalises(int M, int K) { return M <= kFewRows && norm_smem(M, K) <= kNormSmem; }

int launch_gemm_few(cerb_ctx* c, const void* X, const void* W, float* out, int M, int N, int K, cudaStream_t st, const GemmEpilogue* epi,
                    const GemmNorm* norm, unsigned long long* clock_slot) {
  if (M < 1 || M > kFewRows || N < 1 || K < 1 || K % 8 || (((uintptr_t)X | (uintptr_t)W) & 15)) return CERB_E_SHAPE;
  FewParams p;
  memset(&p, 0, sizeof(p));
  p.X = (const bf16*)X;
  p.W = (const bf16*)W;
  p.out = out;
  p.M = M; p.N = N; p.K = K;
  p.clk = clock_slot;
  if (norm) {
    if (!epi || (epi->kind != 1 && epi->kind != 2) || !gemm_few_normalises(M, K)) return CERB_E_SHAPE;
    p.x = norm->x;
    p.gain = (const bf16*)norm->gain;
    p.eps = norm->eps;
  }
  int rc = CERB_E_SHAPE;
  switch (epi ? epi->kind : 0) {
    case 0: rc = launch<0, false>(p, st); break;
    case 1:
      if ((N & 1) || !epi->act) return CERB_E_SHAPE;
      p.F = N / 2;
      p.act = (bf16*)epi->act;
      rc = norm ? launch<1, true>(p, st) : launch<1, false>(p, st);
      break;
    case 2:
      if (!epi->rope || N != 3 * epi->rope->H * 128) return CERB_E_SHAPE;
      p.re = *epi->rope;
      rc = norm ? launch<2, true>(p, st) : launch<2, false>(p, st);
      break;
    case 3:
      if (!epi->x) return CERB_E_SHAPE;
      p.out = epi->x;
      rc = launch<3, false>(p, st);
      break;
  }
  if (rc != CERB_OK) return rc;
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

}  // namespace cerb
