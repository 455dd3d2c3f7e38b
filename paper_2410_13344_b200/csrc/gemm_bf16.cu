// bf16 GEMM of the verification forward on the 5th-generation tensor cores (tcgen05 + TMEM).
//
//   out[slot][m][n] = partial sum over some k range of X[m][k] * W[n][k]        (fp32)
//
// A decoding step has few activation rows (tree nodes x batch) and large weight matrices, so the
// kernel is organised around streaming W exactly once at HBM speed ("swap-AB"): a 128-row tile of
// W is the MMA's A operand (M = 128), the activation rows are the B operand (N = rows), and
// D[128][rows] accumulates in tensor memory and is written out transposed.
//
// 9 to 128 activation rows (gemm_bf16_kernel): a CTA takes 256 weight rows at a time (two MMA tiles
// that share one activation stage), which halves the activation re-reads through L2; weight tiles
// carry an evict-first L2 hint, activation tiles evict-last; the accumulator is double-buffered.
//
// Fewer rows: gemm_few.cu.  More: gemm_tile.cu.
//
// The kernel is launched programmatically dependent on its predecessor: weights do not depend on
// the previous kernel, so the producer fills the whole stage ring with weight tiles before it
// waits for that kernel; only the activation loads and the output stores come after the wait.
//
// Schedule: persistent, one CTA per SM, stream-K.  The work is the list of (weight tile, 64-wide
// k block) units; every CTA takes an equal, contiguous share of it, so all SMs stream for the same
// time whatever the matrix shape (no partial last wave).  A share may cross tile boundaries: each
// run of units inside one tile is a "segment" that accumulates in TMEM and is written to its own
// fp32 partial slot; consumers add a tile's slots in index order (deterministic).  The CTA that
// owns a tile's last segment zero-fills the slots that tile does not use.
//
// Roles inside a CTA (224 threads): warp 0 = TMA producer (one lane) running ahead through the
// whole share, warp 1 = TMEM allocator and MMA issuer (one lane), warp 6 = second MMA issuer,
// warps 2-5 = epilogue (each owns the 32 TMEM lanes of its warp quarter).  The accumulator is double-buffered in TMEM so a segment's
// epilogue overlaps the next segment's MMAs.  Stages and accumulators are handed over with
// mbarriers; every wait is bounded and reports CERB_E_TIMEOUT through a status word.
#include <stdlib.h>
#include <string.h>

#include <mutex>

#include "tc_common.cuh"

namespace cerb {

namespace {

constexpr int BM = 128;          // weight rows per CTA (MMA M)
constexpr int BK = 64;           // k elements per stage: 64 bf16 = one 128-byte swizzle row
constexpr int MAX_STAGES = 8;
constexpr uint32_t A_STAGE_BYTES = BM * BK * 2;

// Loads 16 accumulator columns of this warp's 32 lanes and waits for them.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  tmem_ld16_nowait(taddr, r);
  tmem_ld_wait();
}

struct GemmParams {
  float* out;
  int32_t* status;
  int M, N, K;
  int n_mma;          // activation rows per pass (32..128, power of two)
  int num_kb;         // ceil(K / 64)
  int tiles;          // ceil(N / 128)
  int per;            // work units per CTA
  int total;          // work units in the list: tiles * num_kb
  int nslots;         // partial slots per output element
  int stages;
  long long wait_cycles;   // budget of every bounded wait, SM clock cycles
  uint32_t idesc;
  uint32_t acc_cols;  // TMEM columns of one accumulator buffer
  int tile_rows;      // weight rows between the starts of consecutive tiles
  int half_off;       // weight-row offset of a wide unit's second tile from its first
  unsigned long long* clk;   // measurement only: clk[0] <- min over CTAs of the time the dependency wait returned,
                             // clk[kGemmClockSlots] <- max over CTAs of the time the CTA finished (globaltimer, ns); or null
};

// One run of k blocks inside one (row chunk, weight tile) job.
struct Segment {
  int job, kb0, nkb;
};
__device__ __forceinline__ bool next_segment(int& u, int u1, int num_kb, Segment& sg) {
  if (u >= u1) return false;
  sg.job = u / num_kb;
  sg.kb0 = u - sg.job * num_kb;
  int end = (sg.job + 1) * num_kb;
  if (end > u1) end = u1;
  sg.nkb = end - u;
  u = end;
  return true;
}

__global__ void __launch_bounds__(224, 1) gemm_bf16_kernel(const __grid_constant__ CUtensorMap tmW,
                                                           const __grid_constant__ CUtensorMap tmX, const GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t empty_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t acc_full[2];
  __shared__ __align__(8) uint64_t acc_empty[2];
  __shared__ __align__(8) uint64_t drain_bar[2];       // one per MMA issuer: "everything I issued has retired" (give-up path only)
  __shared__ uint32_t tmem_base_slot;
  __shared__ int aborted_s;
  volatile int* aborted = &aborted_s;
  const WaitCtx wc{p.wait_cycles, aborted, p.status, p.N + 100000 * (p.M > 999 ? 999 : p.M)};

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t b_bytes = (uint32_t)p.n_mma * BK * 2;
  const uint32_t a_bytes = 2 * A_STAGE_BYTES;        // two weight tiles of 128 rows per unit
  const uint32_t stage_bytes = a_bytes + b_bytes;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int share = (int)blockIdx.x;                   // which contiguous share of the unit list
  const int u0 = share * p.per;
  const int u1 = (u0 + p.per < p.total) ? u0 + p.per : p.total;

  if (threadIdx.x == 0) {
    aborted_s = 0;
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 2);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&acc_full[i]), 2);
      mbar_init(smem_u32(&acc_empty[i]), 4);
      mbar_init(smem_u32(&drain_bar[i]), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                 "r"(2u * p.acc_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_slot;

  if (warp == 0) {
    if (lane == 0) {
      const int n_units = u1 - u0;
      const uint64_t pol_w = l2_policy(true), pol_x = l2_policy(false);
      // (tile, k block) of the unit being issued, advanced incrementally
      int w_job = u0 / p.num_kb, w_kb = u0 - w_job * p.num_kb;
      int x_kb = w_kb;
      auto load_w = [&](int i) {
        const int tile = w_job % p.tiles;
        const int s = i % p.stages;
        const uint32_t fb = smem_u32(&full_bar[s]);
        const uint32_t a_dst = smem_base + (uint32_t)s * stage_bytes;
        mbar_expect_tx(fb, stage_bytes);
        tma_load_2d_hint(a_dst, &tmW, w_kb * BK, tile * p.tile_rows, fb, pol_w);
        tma_load_2d_hint(a_dst + A_STAGE_BYTES, &tmW, w_kb * BK, tile * p.tile_rows + p.half_off, fb, pol_w);
        if (++w_kb == p.num_kb) { w_kb = 0; ++w_job; }
      };
      auto load_x = [&](int i) {
        const int s = i % p.stages;
        const uint32_t fb = smem_u32(&full_bar[s]);
        const uint32_t x_dst = smem_base + (uint32_t)s * stage_bytes + a_bytes;
        tma_load_2d_hint(x_dst, &tmX, x_kb * BK, 0, fb, pol_x);
        if (++x_kb == p.num_kb) x_kb = 0;
      };
      // Weights do not depend on the kernel before this one: fill the whole ring with weight tiles
      // while that kernel is still finishing, then wait for it and fetch the activations.
      const int pre = n_units < p.stages ? n_units : p.stages;
      for (int i = 0; i < pre; ++i) load_w(i);
      // the activation map's descriptor is fetched now, not by the first load after the wait
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmX) : "memory");
      griddep_wait();
      // Dependents are released only now, after this CTA's own wait: when the kernel after this one starts,
      // the kernel before this one is complete, which is what lets kernels read, ahead of their own wait,
      // anything written at least two launches earlier.
      griddep_launch();
      if (p.clk) atomicMin(p.clk, globaltimer_ns());
      for (int i = 0; i < pre; ++i) load_x(i);
      int issued = pre;
      for (int i = pre; i < n_units; ++i) {
        const int s = i % p.stages;
        const uint32_t ph = (uint32_t)(i / p.stages) & 1u;
        if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1u, wc, 201)) break;     // this wait gave up (the consumers have stopped): issue nothing more
        load_w(i);
        load_x(i);
        issued = i + 1;
      }
      if (*aborted) {
        // give-up path: the copies already issued still land in this CTA's shared memory; see each of them in
        for (int i = issued > p.stages ? issued - p.stages : 0; i < issued; ++i)
          mbar_wait_drain(smem_u32(&full_bar[i % p.stages]), (uint32_t)(i / p.stages) & 1u);
      }
    }
  } else if (warp == 1 || warp == 6) {
    // MMA issuers.  Issuing one tcgen05.mma occupies its thread for ~100 cycles whatever the MMA's size, and
    // a 64-row step needs eight of them per 32 KB of weights, so each of the two weight tiles of a unit has
    // its own issuing thread (warp 1: first tile, warp 6: second tile).  A stage is free, and an accumulator
    // complete, once both have committed.
    const int hf = warp == 6 ? 1 : 0;
    if (lane == 0) {
      int u = u0;
      Segment sg;
      int i = 0, g = 0;
      while (next_segment(u, u1, p.num_kb, sg)) {
        const int buf = g & 1;
        const uint32_t use = (uint32_t)(g >> 1);      // how often this buffer was used before
        if (!mbar_wait(smem_u32(&acc_empty[buf]), (use & 1u) ^ 1u, wc, 202)) break;
        tc_fence_after();
        const uint32_t tmem_d = tmem_base + (uint32_t)buf * p.acc_cols;
        for (int k = 0; k < sg.nkb; ++k, ++i) {
          int s = i % p.stages;
          uint32_t ph = (uint32_t)(i / p.stages) & 1u;
          if (!mbar_wait(smem_u32(&full_bar[s]), ph, wc, 203)) break;
          tc_fence_after();
          uint32_t a_src = smem_base + (uint32_t)s * stage_bytes;
          uint64_t bdesc = desc_k_sw128(a_src + a_bytes);
          const uint64_t adesc = desc_k_sw128(a_src + (uint32_t)hf * A_STAGE_BYTES);
          const uint32_t d = tmem_d + (uint32_t)(hf * p.n_mma);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)    // advance 16 k elements = 32 bytes inside the swizzled row: +2 in 16-byte units
            umma_bf16(d, adesc + (uint64_t)(kk * 2), bdesc + (uint64_t)(kk * 2), p.idesc, (k > 0 || kk > 0) ? 1u : 0u);
          umma_commit(smem_u32(&empty_bar[s]));     // the stage is free once the MMAs have read it
        }
        if (*aborted) break;
        umma_commit(smem_u32(&acc_full[buf]));       // this thread's part of the segment's accumulator is complete
        ++g;
      }
      if (*aborted) {
        // give-up path: the MMAs already issued still read shared memory and write tensor memory; see them retire
        umma_commit(smem_u32(&drain_bar[hf]));
        mbar_wait_drain(smem_u32(&drain_bar[hf]), 0);
      }
    }
  } else {
    const int quarter = warp & 3;                    // TMEM lanes 32*quarter .. +31 belong to this warp
    griddep_wait();                                  // the kernel before this one may still be reading the partial buffer
    int u = u0;
    Segment sg;
    int g = 0;
    while (next_segment(u, u1, p.num_kb, sg)) {
      const int buf = g & 1;
      const int tile = sg.job;
      if (!mbar_wait(smem_u32(&acc_full[buf]), (uint32_t)(g >> 1) & 1u, wc, 204)) break;                         // the launch's output is undefined from here on
      tc_fence_after();
      // slot = how many CTAs before this one also work on this job
      const int job_u0 = sg.job * p.num_kb;
      const int first_cta = job_u0 / p.per;
      const int last_cta = (job_u0 + p.num_kb - 1) / p.per;
      const int slot = share - first_cta;
      const int m_base = 0;                            // (all rows in one pass: this kernel takes up to 128)
      const int m_cnt = p.M;
      const size_t ldo = (size_t)p.N;
      for (int hf = 0; hf < 2; ++hf) {
        const int n_out = tile * p.tile_rows + hf * p.half_off + quarter * 32 + lane;
        const bool n_ok = n_out < p.N;
        // consecutive lanes hold consecutive output columns: every store instruction writes 128 contiguous bytes
        float* o = p.out + ((size_t)slot * p.M + m_base) * ldo + (n_ok ? n_out : 0);
        const uint32_t taddr = tmem_base + (uint32_t)buf * p.acc_cols + (uint32_t)(hf * p.n_mma) + ((uint32_t)(quarter * 32) << 16);
        for (int c0 = 0; c0 < m_cnt; c0 += 16) {
          uint32_t r[16];
          tmem_ld16(taddr + (uint32_t)c0, r);
          if (n_ok) {
            if (c0 + 16 <= m_cnt) {
#pragma unroll
              for (int j = 0; j < 16; ++j) { *o = __uint_as_float(r[j]); o += ldo; }
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (c0 + j < m_cnt) { *o = __uint_as_float(r[j]); o += ldo; }
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&acc_empty[buf]));
      if (share == last_cta) {
        for (int hf = 0; hf < 2; ++hf) {
          const int n_out = tile * p.tile_rows + hf * p.half_off + quarter * 32 + lane;
          if (n_out >= p.N) continue;
          for (int z = last_cta - first_cta + 1; z < p.nslots; ++z) {
            float* zo = p.out + ((size_t)z * p.M + m_base) * ldo + n_out;
            for (int m = 0; m < m_cnt; ++m) { *zo = 0.f; zo += ldo; }
          }
        }
      }
      ++g;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (p.clk && threadIdx.x == 0) atomicMax(p.clk + kGemmClockSlots, globaltimer_ns());
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(2u * p.acc_cols) : "memory");
  }
}


struct GemmPlan {
  int tiles, num_kb, per, ctas, nslots;
  long long total;   // checked to fit 31 bits before launch
};

// `jobs` x num_kb units cut into `workers` equal contiguous shares.
void cut_shares(GemmPlan& g, long long jobs, int workers) {
  g.total = jobs * g.num_kb;
  long long per = (g.total + workers - 1) / workers;
  int min_per = g.num_kb < 4 ? g.num_kb : 4;          // do not shred tiny problems into one-block segments
  if (per < min_per) per = min_per;
  g.per = (int)per;
  g.ctas = (int)((g.total + per - 1) / per);
  g.nslots = 1;
  for (long long job = 0; job < jobs; ++job) {
    int first = (int)(job * g.num_kb / per), last = (int)((job * g.num_kb + g.num_kb - 1) / per);
    if (last - first + 1 > g.nslots) g.nslots = last - first + 1;
  }
}

// Up to 128 rows: single CTAs, one pass over all rows; a unit is two weight tiles of 128 rows.
GemmPlan make_plan(int sm_count, int N, int K) {
  GemmPlan g;
  g.tiles = (N + 2 * BM - 1) / (2 * BM);
  g.num_kb = (K + BK - 1) / BK;
  cut_shares(g, g.tiles, sm_count);
  return g;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn g_encode = nullptr;

// A box row is 128 bytes (64 bf16); with 256-byte L2 promotion the memory side fetches the neighbouring 128
// bytes of every row as well, i.e. the next (or previous) k block of the same rows, which the same CTA asks
// for right afterwards: DRAM bursts twice as long.  Measured on the 7B decoding step: 4.23 -> 4.02 ms per
// 64-node forward, 3.49 -> 3.31 ms per one-node forward (128-byte promotion and none are equal).

// The last descriptors made, by their arguments.  A descriptor depends on nothing else, and the stand-alone entry
// points (which own no context to keep maps in) are typically called again and again on the same buffers: they
// find their maps here instead of encoding two to six of them per call.
struct MapKey {
  const void* base;
  uint64_t inner, outer, row_bytes;
  uint32_t box_inner, box_outer;
  bool operator==(const MapKey& o) const {
    return base == o.base && inner == o.inner && outer == o.outer && row_bytes == o.row_bytes && box_inner == o.box_inner &&
           box_outer == o.box_outer;
  }
};
constexpr int kMapCache = 32;
std::mutex g_map_mutex;
MapKey g_map_key[kMapCache];
CUtensorMap g_map_val[kMapCache];
int g_map_used = 0, g_map_next = 0;

int encode_2d(CUtensorMap* out, const void* base, uint64_t inner, uint64_t outer, uint64_t row_bytes, uint32_t box_inner,
              uint32_t box_outer) {
  if (init_driver_api() != CERB_OK) return CERB_E_CUDA;
  if (((uintptr_t)base & 15) || (row_bytes & 15)) return CERB_E_SHAPE;
  const MapKey key{base, inner, outer, row_bytes, box_inner, box_outer};
  {
    std::lock_guard<std::mutex> lock(g_map_mutex);
    for (int i = 0; i < g_map_used; ++i)
      if (g_map_key[i] == key) {
        *out = g_map_val[i];
        return CERB_OK;
      }
  }
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {row_bytes};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = g_encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return CERB_E_CUDA;
  std::lock_guard<std::mutex> lock(g_map_mutex);
  g_map_key[g_map_next] = key;
  g_map_val[g_map_next] = *out;
  g_map_next = (g_map_next + 1) % kMapCache;
  if (g_map_used < kMapCache) ++g_map_used;
  return CERB_OK;
}

}  // namespace

int init_driver_api() {
  if (g_encode) return CERB_OK;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess || !fn ||
      q != cudaDriverEntryPointSuccess)
    return CERB_E_CUDA;
  g_encode = (EncodeTiledFn)fn;
  return CERB_OK;
}

int make_weight_map(CUtensorMap* out, const void* W, int N, int K) {
  return encode_2d(out, W, (uint64_t)K, (uint64_t)N, (uint64_t)K * 2, BK, BM);
}

namespace {
// Weight rows [N][K] seen as an array of blocks of rows, so that one box gathers 128 rows in another order.
int encode_rows_nd(CUtensorMap* out, const void* W, int K, int nd, const cuuint64_t* counts, const cuuint64_t* row_strides, const cuuint32_t* box_rows) {
  if (init_driver_api() != CERB_OK) return CERB_E_CUDA;
  if (((uintptr_t)W & 15) || ((size_t)K * 2 & 15)) return CERB_E_SHAPE;
  cuuint64_t dims[5] = {(cuuint64_t)K}, strides[4];
  cuuint32_t box[5] = {BK}, estr[5] = {1, 1, 1, 1, 1};
  for (int i = 0; i < nd; ++i) {
    dims[i + 1] = counts[i];
    strides[i] = row_strides[i] * (cuuint64_t)K * 2;
    box[i + 1] = box_rows[i];
  }
  CUresult r = g_encode(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, nd + 1, const_cast<void*>(W), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? CERB_OK : CERB_E_CUDA;
}
}  // namespace

// [gate rows F][up rows F]: a box is 4 x (16 gate rows, the 16 up rows of the same features).  F a multiple of 16.
int make_gate_up_map(CUtensorMap* out, const void* W, int F, int K) {
  const cuuint64_t counts[3] = {16, 2, (cuuint64_t)F / 16}, strides[3] = {1, (cuuint64_t)F, 16};
  const cuuint32_t box[3] = {16, 2, 4};
  return encode_rows_nd(out, W, K, 3, counts, strides, box);
}

// `heads` blocks of 128 rows: a box is one block as 4 x (rows 16 q .. 16 q + 15, rows 64 + 16 q .. 64 + 16 q + 15).
int make_rotation_map(CUtensorMap* out, const void* W, int heads, int K) {
  const cuuint64_t counts[4] = {16, 2, 4, (cuuint64_t)heads}, strides[4] = {1, 64, 16, 128};
  const cuuint32_t box[4] = {16, 2, 4, 1};
  return encode_rows_nd(out, W, K, 4, counts, strides, box);
}

int make_rows_map(CUtensorMap* out, const void* W, int N, int K, int rows) {
  return encode_2d(out, W, (uint64_t)K, (uint64_t)N, (uint64_t)K * 2, BK, (uint32_t)rows);
}

// The same matrices as tiles of gemm_rows.cu: boxes of `groups` x (4 gate rows, the 4 up rows of the same features) ...
int make_gate_up_groups(CUtensorMap* out, const void* W, int F, int K, int groups) {
  const cuuint64_t counts[3] = {4, 2, (cuuint64_t)F / 4}, strides[3] = {1, (cuuint64_t)F, 4};
  const cuuint32_t box[3] = {4, 2, (cuuint32_t)groups};
  return encode_rows_nd(out, W, K, 3, counts, strides, box);
}

// ... and of `groups` heads x (4 rows of the first half of the head, the same of its second half).
int make_rotation_groups(CUtensorMap* out, const void* W, int heads, int K, int groups) {
  const cuuint64_t counts[3] = {64, 2, (cuuint64_t)heads}, strides[3] = {1, 64, 128};
  const cuuint32_t box[3] = {4, 2, (cuuint32_t)groups};
  return encode_rows_nd(out, W, K, 3, counts, strides, box);
}

int make_act_map(ActMaps* out, const void* X, int rows_alloc, int K, int box_rows) {
  return encode_2d(&out->m[box_rows / 16 - 1], X, (uint64_t)K, (uint64_t)rows_alloc, (uint64_t)K * 2, BK, (uint32_t)box_rows);
}

int make_act_maps(ActMaps* out, const void* X, int rows_alloc, int K) {
  for (int rows = 16; rows <= BM; rows += 16) CERB_TRY(make_act_map(out, X, rows_alloc, K, rows));
  return CERB_OK;
}

// 2-D map over one layer's KV pool viewed as [pages*H*16 rows][Dh]: a box is one page of one head,
// 64 elements (128 bytes) wide.
int make_pool_map(CUtensorMap* out, const void* pool, int n_pool_pages, int H, int Dh) {
  return encode_2d(out, pool, (uint64_t)Dh, (uint64_t)n_pool_pages * H * CERB_PAGE, (uint64_t)Dh * 2, 64, CERB_PAGE);
}

// Number of partial slots the schedule produces for this problem (what consumers must sum).
int gemm_plan_split(int sm_count, int M, int N, int K) {
  return M > BM ? 1 : make_plan(sm_count, N, K).nslots;
}

Chains gemm_bf16_chains(int N, int K) {
  const GemmPlan g = make_plan(148, N, K);
  Chains c;
  for (long long u = 0; u < g.total;) {
    const long long share = (u / g.per + 1) * g.per, job = (u / g.num_kb + 1) * g.num_kb, end = share < job ? share : job;
    c.chain((int)((end < g.total ? end : g.total) - u));
    u = end;
  }
  return c;
}

// Slots of M x N floats that the scratch of the stand-alone GEMM holds.  Up to 128 rows the slots of the plan.  Above, the
// size that callers of that entry have been told to provide: the slots of 74 workers walking 512 weight rows at a time,
// side by side on chunks of 256 rows; the tile plan (gemm_tile.cu) is fitted into it.
int gemm_scratch_slots(int M, int N, int K) {
  GemmPlan g = make_plan(148, N, K);
  if (M <= BM) return g.nslots;
  const int tiles = (N + 4 * BM - 1) / (4 * BM), chunks = (M + kGemmRowsPerPass - 1) / kGemmRowsPerPass;
  const bool grouped = chunks > 1 && chunks * 2 <= 74;
  cut_shares(g, grouped ? tiles : (long long)tiles * chunks, grouped ? 74 / chunks : 74);
  return g.nslots;
}

int launch_gemm_bf16(cerb_ctx* c, const CUtensorMap* tmW, const ActMaps* tmX, float* out, int M, int N, int K,
                     int nsplit, int32_t* status, cudaStream_t st, unsigned long long* clock_slot) {
  if (M <= 0 || N <= 0 || K <= 0 || (K % 8) != 0) return CERB_E_SHAPE;
  if (M > BM) return CERB_E_SHAPE;             // (gemm_tile.cu)
  // Fewer SMs than planned for would need more slots than the caller sized: plan with the number
  // the caller used (148) and simply run that many CTAs; the hardware queues what does not fit.
  GemmPlan g = make_plan(148, N, K);
  if (g.nslots != nsplit) return CERB_E_ARG;
  GemmParams p;
  memset(&p, 0, sizeof(p));
  p.out = out;
  p.status = status;
  p.M = M; p.N = N; p.K = K;
  p.n_mma = row_bucket(M);
  p.num_kb = g.num_kb;
  p.tiles = g.tiles;
  p.per = g.per;
  if (g.total >= (1ll << 30)) return CERB_E_SHAPE;
  p.total = (int)g.total;
  p.nslots = g.nslots;
  p.tile_rows = 2 * BM;
  p.wait_cycles = wait_cycles();
  p.half_off = BM;
  p.clk = clock_slot;
  uint32_t stage_bytes = 2 * A_STAGE_BYTES + (uint32_t)p.n_mma * BK * 2;
  p.stages = (int)((216u * 1024u) / stage_bytes);
  if (p.stages > MAX_STAGES) p.stages = MAX_STAGES;
  if (p.stages < 2) return CERB_E_SHAPE;
  p.acc_cols = 2u * (uint32_t)p.n_mma;            // two weight tiles side by side (at least 32 columns)
  // instruction descriptor: D fp32, A and B bf16, both K-major, N = n_mma, M = 128
  p.idesc = idesc_bf16(BM, (uint32_t)p.n_mma, false, false);
  size_t smem = (size_t)p.stages * stage_bytes + 1024;
  if (smem < 120 * 1024) smem = 120 * 1024;    // one CTA per SM: a CTA may then own all of tensor memory
  static std::atomic<bool> configured{false};
  if (!configured) {
    CERB_CUDA_OK(cudaFuncSetAttribute(gemm_bf16_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(220 * 1024)));
    configured = true;
  }
  if (launch_pdl(gemm_bf16_kernel, dim3(g.ctas), dim3(224), smem, st, *tmW, tmX->box(p.n_mma), p) != cudaSuccess) return CERB_E_CUDA;
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

}  // namespace cerb
