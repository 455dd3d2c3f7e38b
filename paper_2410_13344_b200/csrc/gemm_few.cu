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
// 7B shape, 16 layers and LM head, 1000 tokens before, us per forward of 1 / 2 / 4 / 8 / 12 rows: 1410 / 1381 / 1551 / 1797 /
// 1881; with tensor-memory tiles of 256 weight rows, partial sums in slots and a norm kernel of its own 1664 / 1654 / 1815 /
// 2138 / 2149.  Warps that take k blocks in turn instead of an eighth each: 1436 with one row.
#include <string.h>

#include "cerb_internal.cuh"

namespace cerb {

namespace {

constexpr int WARPS = 8;

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

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mma_16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// KIND as in GemmEpilogue.  NT: column tiles of eight activation rows; KG warps to a row group; U: k blocks of a round; MB CTAs
// to an SM.  The 16 rows of a group are 16 neighbours (0, 3), or eight and the eight that belong to them (1: gate, up; 2:
// elements i and i + 64 of a head).
template <int KIND, int NT, int KG, int U, int MB, bool XB, bool NORM>
__global__ void __launch_bounds__(WARPS * 32, MB) gemm_few_kernel(const __grid_constant__ FewParams p) {
  constexpr bool PAIRS = KIND == 1 || KIND == 2;
  constexpr int RG = WARPS / KG, ROWS = 16 * RG, LD = 8 * NT + 1, ROUND = 32 * U;
  constexpr int OUTS = PAIRS ? ROWS / 2 : ROWS, ITEMS = (OUTS * 8 * NT + WARPS * 32 - 1) / (WARPS * 32);
  __shared__ float red_s[2][KG * ROWS * LD];                 // [tile's parity][k group][row][column + 1]
  extern __shared__ __align__(16) bf16 xs[];                 // NORM: the normalised rows, then the gains; [.][K + 32]
  const int kg = (threadIdx.x >> 5) % KG, rg = (threadIdx.x >> 5) / KG, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int K = p.K;
  // a tile's first row (of a pair: its first member)
  auto first_row = [](int tile) { return KIND == 2 ? (tile / (64 / OUTS)) * 128 + (tile % (64 / OUTS)) * OUTS : tile * OUTS; };
  const bf16* Wr[2];
  const int k0 = kg * p.range + t * 8, k1 = min(K, (kg + 1) * p.range);     // this warp's part of k
  int load_tile = blockIdx.x, load_k = k0;                   // what the next load_w fetches
  auto set_rows = [&]() {
    const int r0 = first_row(load_tile) + (PAIRS ? 8 : 16) * rg + g;
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
  auto load_x = [&](uint4 (&r)[U][NT], int k) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        r[u][n] = make_uint4(0, 0, 0, 0);
        if (k + u * 32 < k1 && 8 * n + g < p.M)
          r[u][n] = NORM ? *reinterpret_cast<const uint4*>(xs + (8 * n + g) * (K + 32) + k + u * 32)
                         : *reinterpret_cast<const uint4*>(p.X + (size_t)(8 * n + g) * K + k + u * 32);
      }
  };
  // (two accumulators in turn: the tensor cores cut the sum off at every step, so half the steps is half the error)
  float acc[2][NT][4];
  auto multiply = [&](const uint4 (&a)[U][2], const uint4 (&x)[U][NT]) {
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        mma_16816(acc[0][n], a[u][0].x, a[u][1].x, a[u][0].y, a[u][1].y, x[u][n].x, x[u][n].y);
        mma_16816(acc[1][n], a[u][0].z, a[u][1].z, a[u][0].w, a[u][1].w, x[u][n].z, x[u][n].w);
      }
  };
  // (XB: X is fetched along with the weights.  Sixteen rows of it leave no registers for that; it comes from L1 or L2 then.)
  uint4 w0[U][2], w1[U][2], x0[U][NT], x1[U][NT];
  set_rows();
  load_w(w0);
  load_k += ROUND;
  load_w(w1);
  if constexpr (NORM)
    for (int j = threadIdx.x * 4; j < K; j += WARPS * 32 * 4)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(xs + p.M * (K + 32) + j)), "l"(p.gain + j) : "memory");
  griddep_wait();
  if (p.clk && threadIdx.x == 0) atomicMin(p.clk, now_ns());
  griddep_launch();
  if constexpr (NORM) {
    // every CTA normalises the rows for itself, while its first weights are on their way
    __shared__ float ss_s[8 * NT][WARPS];
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
      if (lane == 0) ss_s[m][threadIdx.x >> 5] = ss;
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
  if (XB) {
    load_x(x0, k0);
    load_x(x1, k0 + ROUND);
  }
  int pos[ITEMS], kv[ITEMS];
  if constexpr (KIND == 2) {
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int m = (it * WARPS * 32 + threadIdx.x) / OUTS;
      pos[it] = kv[it] = -1;
      if (m < p.M) {
        const RopeEpilogue& e = p.re;
        int b, v;
        locate_row(m, e.row_off, e.B, e.n, b, v);
        const int at = e.len[b] + e.depth[v], slot = e.len[b] + v;
        if (v < e.n_active[b] && at < e.max_pos && slot < e.max_pos) {
          pos[it] = at;
          kv[it] = e.page_table[(size_t)b * e.max_pages + slot / CERB_PAGE] * e.H * CERB_PAGE + slot % CERB_PAGE;
        }
      }
    }
  }
  int parity = 0;
  for (int tile = blockIdx.x; tile < p.tiles; tile += gridDim.x, parity ^= 1) {
    const int first = first_row(tile);
    float old[ITEMS];
    if constexpr (KIND == 3) {
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) {
        const int i = it * WARPS * 32 + threadIdx.x, m = i / OUTS, rr = i % OUTS;
        old[it] = m < p.M && first + rr < p.N ? p.out[(size_t)m * p.N + first + rr] : 0.f;
      }
    }
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[0][n][e] = acc[1][n][e] = 0.f;
    // rounds in pairs (p.rounds of them); the loads run two rounds ahead, over the end of the tile into the next
    for (int q = 0; q < p.rounds; q += 2) {
      const bool last = q + 2 >= p.rounds;
      if (last) {
        load_tile += gridDim.x;
        load_k = k0;
        if (!XB) load_x(x0, k0 + q * ROUND);
        multiply(w0, x0);
        set_rows();
      } else {
        load_k = k0 + (q + 2) * ROUND;
        if (!XB) load_x(x0, k0 + q * ROUND);
        multiply(w0, x0);
      }
      load_w(w0);
      if (XB) load_x(x0, load_k);
      load_k += ROUND;
      if (!XB) load_x(x1, k0 + (q + 1) * ROUND);
      multiply(w1, x1);
      load_w(w1);
      if (XB) load_x(x1, load_k);
    }
    float* red = red_s[parity];
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        red[(kg * ROWS + 16 * rg + 8 * (e >> 1) + g) * LD + 8 * n + 2 * t + (e & 1)] = acc[0][n][e] + acc[1][n][e];
    __syncthreads();
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int i = it * WARPS * 32 + threadIdx.x, m = i / OUTS, rr = i % OUTS;
      if (m >= p.M) continue;
      auto sum = [&](int row) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < KG; ++q) s += red[(q * ROWS + row) * LD + m];
        return s;
      };
      if constexpr (!PAIRS) {
        if (first + rr >= p.N) continue;
        const float s = sum(rr);
        p.out[(size_t)m * p.N + first + rr] = KIND == 3 ? old[it] + s : s;
      } else {
        const int row = 16 * (rr >> 3) + (rr & 7);
        float a = sum(row), b = sum(row + 8);
        if constexpr (KIND == 1) {
          if (first + rr < p.F) p.act[(size_t)m * p.F + first + rr] = __float2bfloat16_rn(a / (1.0f + expf(-a)) * b);
        } else {
          if (kv[it] < 0) continue;
          const RopeEpilogue& e = p.re;
          const int unit = first >> 7, el = (first & 127) + rr, which = unit / e.H, h = unit - which * e.H;
          if (which < 2) {
            const float2 cs = e.rope[(size_t)pos[it] * 64 + el];
            const float o1 = a * cs.x - b * cs.y;
            b = b * cs.x + a * cs.y;
            a = o1;
          }
          bf16* o = which == 0 ? reinterpret_cast<bf16*>(e.q) + ((size_t)m * e.H + h) * 128 + el
                               : reinterpret_cast<bf16*>(which == 1 ? e.kpool : e.vpool) + ((size_t)kv[it] + (size_t)h * CERB_PAGE) * 128 + el;
          o[0] = __float2bfloat16_rn(a);
          o[64] = __float2bfloat16_rn(b);
        }
      }
    }
  }
  if (p.clk && threadIdx.x == 0) atomicMax(p.clk + kGemmClockSlots, now_ns());
}

// Rows whose norm a GEMM computes itself: as many as fit 25 KB of shared memory with the gains, two of 4096 columns.  (One
// row: 1419 us for the forward above instead of 1513 with a norm kernel; eight: 2154 instead of 1793, their rows' loads queue
// behind the weights that every CTA has in flight.)
constexpr size_t kNormSmem = 25 * 1024;
size_t norm_smem(int M, int K) { return (size_t)(M + 1) * (K + 32) * sizeof(bf16); }

template <int KIND, int NT, int KG, int U, int MB, bool XB, bool NORM>
int launch(FewParams p, cudaStream_t st) {
  constexpr int ROWS = 16 * (WARPS / KG), OUTS = KIND == 1 || KIND == 2 ? ROWS / 2 : ROWS, ROUND = 32 * U;
  p.tiles = ((KIND == 1 ? p.F : KIND == 2 ? p.N / 2 : p.N) + OUTS - 1) / OUTS;
  p.rounds = (p.K + KG * ROUND - 1) / (KG * ROUND);
  p.range = p.rounds * ROUND;
  p.rounds = (p.rounds + 1) & ~1;
  const int grid = p.tiles < 148 * MB ? p.tiles : 148 * MB;
  auto kern = gemm_few_kernel<KIND, NT, KG, U, MB, XB, NORM>;
  const size_t smem = NORM ? norm_smem(p.M, p.K) : 0;
  static bool configured = false;
  if (!configured) {
    // the share of the SM's memory that MB CTAs need as shared memory; the rest is L1
    constexpr size_t most = NORM ? kNormSmem : 0;
    const int share = (int)((MB * (2 * KG * ROWS * (8 * NT + 1) * sizeof(float) + most + 1024) * 100 + 228 * 1024 - 1) / (228 * 1024));
    if (NORM) CERB_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kNormSmem));
    CERB_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, share));
    configured = true;
  }
  return launch_pdl(kern, dim3(grid), dim3(WARPS * 32), smem, st, p) == cudaSuccess ? CERB_OK : CERB_E_CUDA;
}

template <int KIND>
int pick(const FewParams& p, cudaStream_t st) {
  if constexpr (KIND == 1 || KIND == 2) {
    if (p.x) return launch<KIND, 1, 8, 4, 2, true, true>(p, st);
  }
  return p.M <= 8 ? launch<KIND, 1, 8, 4, 2, true, false>(p, st) : launch<KIND, 2, 8, 4, 2, false, false>(p, st);
}

}  // namespace

bool gemm_few_normalises(int M, int K) { return M <= 8 && norm_smem(M, K) <= kNormSmem; }

int launch_gemm_few(const void* X, const void* W, float* out, int M, int N, int K, cudaStream_t st, const GemmEpilogue* epi,
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
  switch (epi ? epi->kind : 0) {
    case 0: return pick<0>(p, st);
    case 1:
      if ((N & 1) || !epi->act) return CERB_E_SHAPE;
      p.F = N / 2;
      p.act = (bf16*)epi->act;
      return pick<1>(p, st);
    case 2:
      if (!epi->rope || N != 3 * epi->rope->H * 128) return CERB_E_SHAPE;
      p.re = *epi->rope;
      return pick<2>(p, st);
    case 3:
      if (!epi->x) return CERB_E_SHAPE;
      p.out = epi->x;
      return pick<3>(p, st);
  }
  return CERB_E_SHAPE;
}

}  // namespace cerb
