// bf16 GEMM for more than 128 activation rows (batched trees, prefill): output tiles on CTA pairs (tcgen05 cta_group::2).
//
//   D[256 HF weight rows][up to 256 activation rows] per tile, fp32, in the tensor memory of two CTAs, HF = 1 or 2
//
// What bounds it: the tensor pipe and the power limit from about 1000 rows on, L2 (11.6 TB/s measured on the way to the
// SMs) at a few hundred rows, the weight stream at 256 rows and fewer.
//
// Tile.  One MMA is 256 weight rows tall, 128 from each CTA's shared memory, and its activation rows (the MMA's N, up to
// 256) come half from each CTA; each CTA's tensor memory receives its 128 rows of D.  An accumulator takes up to 256 of the
// 512 columns.
//   HF = 1: one accumulator per tile, so there are two of them and a tile's epilogue runs under the next tile's MMAs.
//           With few tiles per pair they hold the even and the odd k blocks of one tile instead (`chains`): a chain of
//           tensor-core accumulations loses about half a unit in the last place per step, always towards zero, and 4096 k in
//           one chain doubled the share of bf16 results that round the other way (keys of the first layer at the 13B width
//           against the oracle, mean difference: 3.0e-6 in chains of up to 33 k blocks, 6.9e-6 in chains of 80).
//           Where the fp32 product itself is the result (KIND 0) a chain is `fill` k blocks long: then the other accumulator
//           goes on, and the epilogue warps add what is there to their registers.  Relative error (2-norm, against float64)
//           of 4096 k: 4.4e-6 in one chain, 2.1e-6 in two, 1.0e-6 in fills of 16 and 0.5e-6 of 8.  Taking a fill over costs
//           the warps 3.4 us, of which the last one shows (256 x 12288 x 4096: 36 us in one chain, 40 in fills of 16, 46 of 8).
//   HF = 2: two MMA rows share one activation tile: 96 KB instead of 128 KB from L2 per 512 x 256 x 64, but the epilogue is
//           covered only as far as the MMAs of the next tile's first accumulator run under the second one's.
// A stage is 64 k.  M rows are cut into equal chunks of up to 256, rounded up to 32 rows.
//
// Schedule (make_tile_plan chooses by a cost model).  Every output has one sum, written once by an epilogue:
//   - whole tiles dealt out in turn; neighbouring pairs work on the chunks of one weight tile, so HBM delivers it once;
//   - few tiles: S pairs per tile, each a range of k.  Every pair leaves the columns that others finish in a fix-up buffer
//     and finishes its own share of them, adding the others' sums in k order (a reduce-scatter through L2);
//   - a last wave that would be nearly empty, or fewer tiles than pairs: up to two tiles per pair are cut along k into equal
//     shares, which are done first.  Of the pairs that meet in a tile the last one to finish its run adds up what the others
//     have left in the fix-up buffer, in k order, and runs the epilogue.
// Pairs that wait for one another get on whatever else holds SMs.  With shares, the one that waits is the last: the others are
// already writing what it waits for.  With S pairs to a tile they have neighbouring block indices and no other tile, so of
// those resident at any time only the ones of the last tile begun can be waiting for pairs that are not.  (A pair must not
// be given a second tile there, nor the pairs of a tile be spread out.)
//
// Epilogues (KIND; 0 writes the product):
//   1  SwiGLU.  The weight tile is fetched with 16 gate rows and the 16 up rows of the same features in turn (a 4-D view
//      of the matrix), so a warp's 32 accumulator lanes hold 16 (gate, up) pairs; one shuffle per two columns brings the
//      members of a pair together, and half a warp finishes one activation row, the other half the next.
//   2  RoPE and cache append (head_dim 128).  A CTA's 128 weight rows are one head of q, k or v, fetched so that elements i
//      and i + 64 of a rotation pair sit 16 lanes apart (a 5-D view).  Arithmetic and order as in rope_append_kernel.
//   3  Residual add: the tile is added to the fp32 residual stream.
// They replace passes of element-wise kernels over the fp32 sums.
#include <math.h>
#include <string.h>

#include <type_traits>

#include "tc_common.cuh"

namespace cerb {

namespace {

constexpr int BK = 64;
constexpr int MAX_STAGES = 8;
constexpr int TILE_X = kGemmRowsPerPass;                   // activation rows of a tile at most
constexpr uint32_t A_BYTES = 128 * BK * 2;
constexpr int kPairs = 74;
constexpr int COLS = 16;                                   // columns an epilogue warp takes at a time
constexpr int kEpiWarps = 16;                              // four per 32 tensor-memory lanes
constexpr int kThreads = 64 + 32 * kEpiWarps;

struct TileParams {
  float* out;               // KIND 0: [M][N]; KIND 3: the residual stream [M][N]
  float* fix;               // [pair][its first, its last run in a cut tile][CTA][accumulator][column / 4][128 lanes][4]; S > 1: no heads
  unsigned int* tickets;    // [split tile][CTA][epilogue warp], zero on entry and on exit
  bf16* act;                // KIND 1: [M][F]
  RopeEpilogue re;          // KIND 2
  int32_t* status;
  int M, N, F;
  int n_act;                // activation rows per chunk
  int stages;
  int mchunks, num_kb, tiles;
  int chains;                    // 2 (HF = 1): the two accumulators hold the even and the odd k blocks of a tile
  int fill;                      // KIND 0: k blocks that an accumulator takes before its sums move to registers
  int S;                         // pairs per tile
  int sk_tiles, per, sk_total;   // tiles cut along k into equal shares, k blocks per share, k blocks in all of them
  long long wait_cycles;
  unsigned long long* clk;
};

// A run of k blocks inside one tile.
struct Run {
  int tile, kb0, nkb;
};
struct Work {
  int u, u1, whole, step, tiles, num_kb, S, part;
  __device__ __forceinline__ Work(const TileParams& p, int pair, int pairs)
      : u(pair * p.per), u1(min(pair * p.per + p.per, p.sk_total)), whole(p.S > 1 ? pair / p.S : p.sk_tiles + pair), step(pairs), tiles(p.tiles),
        num_kb(p.num_kb), S(p.S), part(pair % p.S) {}
  __device__ __forceinline__ bool next(Run& r) {
    if (u < u1) {
      r.tile = u / num_kb;
      r.kb0 = u - r.tile * num_kb;
      r.nkb = min((r.tile + 1) * num_kb, u1) - u;
      u += r.nkb;
      return true;
    }
    if (whole >= tiles) return false;
    r.tile = whole;
    r.kb0 = part * num_kb / S;
    r.nkb = (part + 1) * num_kb / S - r.kb0;
    whole += step;
    return true;
  }
};

// Position in the stage ring and the parity of its current round.
struct Ring {
  int s = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next(int stages) {
    if (++s == stages) { s = 0; ph ^= 1u; }
  }
};

template <int KIND>
__device__ __forceinline__ void load_weights(uint32_t dst, const CUtensorMap* map, int kb, int unit, uint32_t bar, uint64_t pol) {
  const int x = kb * BK;
  if constexpr (KIND == 1)
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
        ::"r"(dst), "l"((uint64_t)map), "r"(x), "r"(0), "r"(0), "r"(unit * 4), "r"(bar), "l"(pol)
        : "memory");
  else if constexpr (KIND == 2)
    asm volatile(
        "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5, %6}], [%7], %8;"
        ::"r"(dst), "l"((uint64_t)map), "r"(x), "r"(0), "r"(0), "r"(0), "r"(unit), "r"(bar), "l"(pol)
        : "memory");
  else
    tma_load_2d_pair(dst, map, x, unit * 128, bar, pol);
}

// Finishes 16 columns (activation rows row0 + c0 ...) of one accumulator lane.  What an epilogue costs is latency: everything
// is computed before anything is stored (with the bounds checks of the stores in between, each column's chain came after the
// last one's: QKV of the 7B shape at 512 rows 103 us instead of 58), and sixteen warps with 16 columns each take turns
// (eight with 32: 22 us for the two accumulators of a 512-row SwiGLU tile whose MMAs take 37).
template <int KIND>
__device__ __forceinline__ void finish(const TileParams& p, const float* v, int unit, int quarter, int lane, int row0, int c0,
                                       const int* pos_s, const int* kv_s) {
  const int left = min(COLS, min(p.n_act - c0, p.M - row0 - c0));          // live columns
  if constexpr (KIND == 0 || KIND == 3) {
    const int n_out = unit * 128 + quarter * 32 + lane;
    if (n_out >= p.N) return;
    float* o = p.out + (size_t)(row0 + c0) * p.N + n_out;     // (consecutive lanes: consecutive columns of a row)
    float x[COLS];
#pragma unroll
    for (int j = 0; j < COLS; ++j) x[j] = KIND == 3 && j < left ? o[(size_t)j * p.N] : 0.f;
    if (left == COLS) {
#pragma unroll
      for (int j = 0; j < COLS; ++j) o[(size_t)j * p.N] = KIND == 3 ? x[j] + v[j] : v[j];
    } else {
#pragma unroll
      for (int j = 0; j < COLS; ++j)
        if (j < left) o[(size_t)j * p.N] = KIND == 3 ? x[j] + v[j] : v[j];
    }
  } else {
    constexpr int P = COLS / 2;
    const int hi = lane >> 4;
    const int i = quarter * 16 + (lane & 15);                               // feature / rotation index inside the unit
    // lanes 0-15 hold the first member of each pair (gate; element i), lanes 16-31 the second (up; element i + 64):
    // the lower half of the warp finishes column 2 j, the upper half column 2 j + 1
    float a[P], b[P];
#pragma unroll
    for (int j = 0; j < P; ++j) {
      const float got = __shfl_xor_sync(0xffffffffu, hi ? v[2 * j] : v[2 * j + 1], 16);
      a[j] = hi ? got : v[2 * j];
      b[j] = hi ? v[2 * j + 1] : got;
    }
    if constexpr (KIND == 1) {
      const int f = unit * 64 + i;
#pragma unroll
      for (int j = 0; j < P; ++j) a[j] = a[j] / (1.0f + expf(-a[j])) * b[j];
      if (f >= p.F) return;
      bf16* o = p.act + (size_t)(row0 + c0 + hi) * p.F + f;
#pragma unroll
      for (int j = 0; j < P; ++j)
        if (2 * j + hi < left) o[(size_t)(2 * j) * p.F] = __float2bfloat16_rn(a[j]);
    } else {
      if (unit >= 3 * p.re.H) return;
      const int which = unit / p.re.H, h = unit - which * p.re.H;
      int kv[P];
#pragma unroll
      for (int j = 0; j < P; ++j) kv[j] = 2 * j + hi < left ? kv_s[c0 + 2 * j + hi] : -1;
      if (which < 2) {
        float2 cs[P];
#pragma unroll
        for (int j = 0; j < P; ++j) {
          const int pos = pos_s[c0 + 2 * j + hi];
          cs[j] = p.re.rope[(size_t)(pos < 0 ? 0 : pos) * 64 + i];
        }
#pragma unroll
        for (int j = 0; j < P; ++j) {
          const float o1 = a[j] * cs[j].x - b[j] * cs[j].y;
          b[j] = b[j] * cs[j].x + a[j] * cs[j].y;
          a[j] = o1;
        }
      }
      bf16* q = reinterpret_cast<bf16*>(p.re.q) + ((size_t)(row0 + c0 + hi) * p.re.H + h) * 128 + i;
      bf16* pool = reinterpret_cast<bf16*>(which == 1 ? p.re.kpool : p.re.vpool) + (size_t)h * CERB_PAGE * 128 + i;
#pragma unroll
      for (int j = 0; j < P; ++j) {
        bf16* o = which == 0 ? q + (size_t)(2 * j) * p.re.H * 128 : pool + (size_t)kv[j] * 128;
        if (kv[j] >= 0) {
          o[0] = __float2bfloat16_rn(a[j]);
          o[64] = __float2bfloat16_rn(b[j]);
        }
      }
    }
  }
}

// Warp by warp, the pairs that share a tile go by one counter in global memory (bounded wait).
//   shares: each takes a number; all but the last leave their sums in the fix-up buffer and add kFixDone, the last one waits for
//     that and adds them to its own, which have stayed in tensor memory;
//   S pairs: each adds 1 when what it leaves is written, waits for all S, and adds kFixDone when it has read what it needs;
//     the last one to do so puts the counter back to zero.
constexpr unsigned int kFixDone = 256u;
__device__ __forceinline__ unsigned int ld_acquire(const unsigned int* a) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}
__device__ __forceinline__ bool wait_fix(const unsigned int* ticket, unsigned int mask, unsigned int least, const WaitCtx& w, int site) {
  const long long t0 = clock64();
  const long long budget = *w.aborted ? kAbortedWaitCycles : w.budget;
  for (;;) {
    for (int i = 0; i < 16; ++i)
      if ((ld_acquire(ticket) & mask) >= least) return true;
    if (clock64() - t0 > budget) break;
  }
  wait_ran_out(w, site);
  return false;
}

__device__ __forceinline__ void ld_acc(uint32_t taddr, float* v) {
  tmem_ld16_nowait(taddr, reinterpret_cast<uint32_t*>(v));
  tmem_ld_wait();
}
__device__ __forceinline__ void put_fix(float4* at, const float* v) {
#pragma unroll
  for (int j = 0; j < COLS / 4; ++j) __stcg(at + j * 128, make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]));
}
__device__ __forceinline__ void get_fix(const float4* at, float4* o) {
#pragma unroll
  for (int j = 0; j < COLS / 4; ++j) o[j] = __ldcg(at + j * 128);
}
__device__ __forceinline__ void add(const float4* o, float* v) {
#pragma unroll
  for (int j = 0; j < COLS / 4; ++j) { v[4 * j] += o[j].x; v[4 * j + 1] += o[j].y; v[4 * j + 2] += o[j].z; v[4 * j + 3] += o[j].w; }
}

template <int KIND, int HF>
__global__ void __launch_bounds__(kThreads, 1) gemm_tile_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                                                                const TileParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[MAX_STAGES];      // used in the pair's first CTA only
  __shared__ __align__(8) uint64_t empty_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2]; // acc_empty: first CTA only, the epilogue warps of both CTAs arrive
  __shared__ __align__(8) uint64_t drain_bar, meet_bar;
  __shared__ int pos_s[KIND == 2 ? TILE_X : 1], kv_s[KIND == 2 ? TILE_X : 1];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int aborted_s, meet_flag_s;
  volatile int* aborted = &aborted_s;
  const WaitCtx wc{p.wait_cycles, aborted, p.status, p.N + 100000 * (p.M > 999 ? 999 : p.M)};

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t stage_bytes = HF * A_BYTES + (uint32_t)p.n_act * BK;          // (half the chunk's activation rows)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const bool first = rank == 0;
  const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;

  if (threadIdx.x == 0) {
    aborted_s = 0;
    meet_flag_s = 0;
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&acc_full[i]), 1);
      mbar_init(smem_u32(&acc_empty[i]), 2 * kEpiWarps / HF);
    }
    mbar_init(smem_u32(&drain_bar), 1);
    mbar_init(smem_u32(&meet_bar), 2);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    // each CTA allocates all 512 columns of its own tensor memory (so both get the same base)
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_start_arrive();       // the other CTA's barriers exist before anything is signalled across
  cluster_start_wait();
  const uint32_t tmem_base = tmem_base_slot;

  if (warp == 0) {
    if (lane == 0) {
      // weights that several row chunks read, at different times where tiles are cut along k, stay in L2 like anything else
      const uint64_t pol_w = p.mchunks > 1 ? l2_policy_normal() : l2_policy(true), pol_x = l2_policy(false);
      const uint32_t tx = 2u * stage_bytes;                                   // both CTAs' copies of a stage
      Work ww(p, pair, pairs), wx(p, pair, pairs);                           // weights run ahead of activations before the wait
      Run rw, rx;
      rw.nkb = rx.nkb = 0;
      Ring qw, qx;
      auto more_w = [&]() { return rw.nkb > 0 || ww.next(rw); };
      auto load_w = [&]() {
        if (first) mbar_expect_tx(smem_u32(&full_bar[qw.s]), tx);
#pragma unroll
        for (int hf = 0; hf < HF; ++hf)
          load_weights<KIND>(smem_base + (uint32_t)qw.s * stage_bytes + hf * A_BYTES, &tmW, rw.kb0, ((rw.tile / p.mchunks) * HF + hf) * 2 + rank,
                             mapa_u32(smem_u32(&full_bar[qw.s]), 0), pol_w);
        ++rw.kb0;
        --rw.nkb;
        qw.next(p.stages);
      };
      auto load_x = [&]() {
        if (rx.nkb == 0) wx.next(rx);
        tma_load_2d_pair(smem_base + (uint32_t)qx.s * stage_bytes + HF * A_BYTES, &tmX, rx.kb0 * BK, (rx.tile % p.mchunks) * p.n_act + rank * (p.n_act >> 1),
                         mapa_u32(smem_u32(&full_bar[qx.s]), 0), pol_x);
        ++rx.kb0;
        --rx.nkb;
        qx.next(p.stages);
      };
      int issued = 0;
      for (; issued < p.stages && more_w(); ++issued) load_w();
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmX) : "memory");
      griddep_wait();
      griddep_launch();
      if (p.clk) atomicMin(p.clk, globaltimer_ns());
      for (int i = 0; i < issued; ++i) load_x();
      for (; more_w(); ++issued) {
        if (!mbar_wait_cluster(smem_u32(&empty_bar[qw.s]), qw.ph ^ 1u, wc, 221)) break;
        load_w();
        load_x();
      }
      if (*aborted) {
        // give-up path: this CTA's copies land in its own shared memory but are counted on the first CTA's
        // barriers, and the two CTAs may have stopped at different stages, so neither can see exactly its own
        // copies in.  The first CTA waits for the stages it knows of (short budget); then both let the time of
        // many memory round trips pass before they go on to the rendezvous and leave.
        if (first)
          for (int i = issued > p.stages ? issued - p.stages : 0; i < issued; ++i)
            mbar_wait_drain(smem_u32(&full_bar[i % p.stages]), (uint32_t)(i / p.stages) & 1u, 2000000ll);
        const long long t_land = clock64();
        while (clock64() - t_land < 400000ll) __nanosleep(1000);
      }
    }
  } else if (warp == 1) {
    // MMA issuer of the pair (first CTA).  The whole warp walks the list and one elected lane issues.
    if (first) {
      const uint32_t idesc = idesc_bf16(256, (uint32_t)p.n_act, false, false);
      Work w(p, pair, pairs);
      Run r;
      Ring q0, q;                        // stage of the next MMAs of the first / of the last accumulator
      bool live = true;
      auto wait = [&](uint64_t& bar, uint32_t parity, int site) {
        const bool ok = mbar_wait_cluster(smem_u32(&bar), parity, wc, site);
        live = __all_sync(0xffffffffu, ok);
        tc_fence_after();
        return live;
      };
      auto issue = [&](int stage, int hf, uint32_t d, bool fresh) {
        const uint32_t src = smem_base + (uint32_t)stage * stage_bytes;
        const uint64_t adesc = desc_k_sw128(src + hf * A_BYTES), bdesc = desc_k_sw128(src + HF * A_BYTES);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk)
          umma_bf16_pair(d, adesc + (uint64_t)(kk * 2), bdesc + (uint64_t)(kk * 2), idesc, (!fresh || kk > 0) ? 1u : 0u);
      };
      for (int g = 0; live && w.next(r);) {
        if constexpr (HF == 1) {
          const bool two = p.chains == 2;
          const int fill = KIND == 0 ? p.fill : r.nkb;
          for (int left = r.nkb; live && left > 0; left -= fill, ++g) {
            const int buf = two ? 0 : g & 1, n = min(fill, left);
            if (!wait(acc_empty[buf], ((uint32_t)(two ? g : g >> 1) & 1u) ^ 1u, 222)) break;
            for (int k = 0; k < n; ++k) {
              if (!wait(full_bar[q.s], q.ph, 223)) break;
              if (elect_one()) {
                issue(q.s, 0, tmem_base + (uint32_t)((two ? k & 1 : buf) * TILE_X), k < p.chains);
                umma_commit_pair(smem_u32(&empty_bar[q.s]));       // the stage is free in both CTAs once these MMAs have read it
                if (k + 1 == n) umma_commit_pair(smem_u32(&acc_full[buf]));
              }
              __syncwarp();
              q.next(p.stages);
            }
          }
        } else {
          const uint32_t free_ph = ((uint32_t)g & 1u) ^ 1u;
          if (!wait(acc_empty[0], free_ph, 222)) break;
          // while the second accumulator of the tile before is still being read out, the first one runs ahead
          int n0 = 0;
          const int ahead = min(r.nkb, p.stages);
          while (n0 < ahead && !__all_sync(0xffffffffu, mbar_try_wait_cluster(smem_u32(&acc_empty[1]), free_ph))) {
            if (!wait(full_bar[q0.s], q0.ph, 223)) break;
            if (elect_one()) {
              issue(q0.s, 0, tmem_base, n0 == 0);
              if (n0 + 1 == r.nkb) umma_commit_pair(smem_u32(&acc_full[0]));
            }
            __syncwarp();
            q0.next(p.stages);
            ++n0;
          }
          if (!live || !wait(acc_empty[1], free_ph, 227)) break;
          for (int k = 0; k < r.nkb; ++k) {
            if (k >= n0 && !wait(full_bar[q.s], q.ph, 223)) break;
            if (elect_one()) {
              if (k >= n0) {
                issue(q.s, 0, tmem_base, k == 0);
                if (k + 1 == r.nkb) umma_commit_pair(smem_u32(&acc_full[0]));
              }
              issue(q.s, 1, tmem_base + TILE_X, k == 0);
              umma_commit_pair(smem_u32(&empty_bar[q.s]));
              if (k + 1 == r.nkb) umma_commit_pair(smem_u32(&acc_full[1]));
            }
            __syncwarp();
            q.next(p.stages);
          }
          q0 = q;
          ++g;
        }
      }
      if ((!live || *aborted) && elect_one()) {            // (an issuer whose own waits hold ends like the others, too)
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&drain_bar)) : "memory");
        mbar_wait_drain(smem_u32(&drain_bar), 0, 40000000ll);
      }
    }
  } else {
    const int quarter = warp & 3;                    // tensor-memory lanes 32 * quarter .. + 31 belong to this warp
    const int ew = warp - 2;
    // which blocks of columns: HF = 1: every fourth; HF = 2: of the first or of the second accumulator, every second
    const int hf = HF == 2 ? ew >> 3 : 0;
    const int c_first = (HF == 2 ? (ew >> 2) & 1 : ew >> 2) * COLS;
    constexpr int C_STEP = HF == 2 ? 2 * COLS : 4 * COLS;
    const int et = quarter * 32 + lane;
    griddep_wait();                                  // the kernels before this one may still be reading what this one writes
    const uint32_t ae[2] = {mapa_u32(smem_u32(&acc_empty[0]), 0), mapa_u32(smem_u32(&acc_empty[1]), 0)};
    Work w(p, pair, pairs);
    Run r;
    int chunk_known = -1;
    // A warp whose wait has run out writes nothing more, but goes through the remaining runs (every later wait is short
    // then): the other epilogue warps meet it at named barriers, other pairs at the counters.
    bool live = true;
    int g = 0;                                       // accumulator fills so far
    while (w.next(r)) {
      const int chunk = r.tile % p.mchunks, row0 = chunk * p.n_act;
      if (KIND == 2 && chunk != chunk_known) {
        // positions and cache rows of the chunk's activation rows
        asm volatile("bar.sync 2, 512;" ::: "memory");                       // (the previous tile's readers are done)
        const RopeEpilogue& e = p.re;
        for (int c = ew * 32 + lane; c < TILE_X; c += 32 * kEpiWarps) {
          int pos = -1, kv = -1;
          if (c < p.n_act && row0 + c < p.M) {
            int b, v;
            locate_row(row0 + c, e.row_off, e.B, e.n, b, v);
            const int at = e.len[b] + e.depth[v], slot = e.len[b] + v;
            if (v < e.n_active[b] && at < e.max_pos && slot < e.max_pos) {
              pos = at;
              kv = e.page_table[(size_t)b * e.max_pages + slot / CERB_PAGE] * e.H * CERB_PAGE + slot % CERB_PAGE;
            }
          }
          pos_s[c] = pos;
          kv_s[c] = kv;
        }
        asm volatile("bar.sync 2, 512;" ::: "memory");
        chunk_known = chunk;
      }
      int first_share = pair, last_share = pair;
      if (r.tile < p.sk_tiles) {
        first_share = r.tile * p.num_kb / p.per;
        last_share = (r.tile * p.num_kb + p.num_kb - 1) / p.per;
      }
      const int parts = last_share - first_share + 1;
      const int unit = ((r.tile / p.mchunks) * HF + hf) * 2 + rank;
      const bool two = HF == 1 && p.chains == 2;
      int acc = hf;                                                          // the accumulator that ends up with the run's sums
      auto filled = [&](int i, uint32_t parity) {
        if (!mbar_wait_cluster(smem_u32(&acc_full[i]), parity, wc, 224)) live = false;      // the output is undefined from here on
        live = __all_sync(0xffffffffu, live);
        tc_fence_after();
      };
      auto release = [&](int i) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(ae[i]);          // (the first CTA's own warps arrive the same way)
      };
      const uint32_t lanes = tmem_base + ((uint32_t)(quarter * 32) << 16);
      if constexpr (HF == 2) {
        filled(hf, (uint32_t)g & 1u);
        ++g;
      } else if (KIND != 0 || r.nkb <= p.fill) {
        acc = two ? 0 : g & 1;
        filled(acc, (uint32_t)(two ? g : g >> 1) & 1u);
        ++g;
      } else {
        // several fills: this warp's columns wait in registers, the last fill's accumulator receives their sum
        constexpr int BLOCKS = TILE_X / C_STEP;
        float held[BLOCKS][COLS];
        for (int left = r.nkb;; left -= p.fill) {
          acc = g & 1;
          filled(acc, (uint32_t)(g >> 1) & 1u);
          ++g;
          const uint32_t from = lanes + (uint32_t)(acc * TILE_X + c_first);
#pragma unroll
          for (int i = 0; i < BLOCKS; ++i)
            if (c_first + i * C_STEP < p.n_act) {
              float v[COLS];
              ld_acc(from + (uint32_t)(i * C_STEP), v);
#pragma unroll
              for (int j = 0; j < COLS; ++j) held[i][j] = left == r.nkb ? v[j] : held[i][j] + v[j];
              if (left <= p.fill) tmem_st16(from + (uint32_t)(i * C_STEP), reinterpret_cast<const uint32_t*>(held[i]));
            }
          if (left <= p.fill) break;
          release(acc);
        }
        tmem_st_wait();
      }
      const uint32_t taddr = lanes + (uint32_t)(acc * TILE_X);
      auto read_acc = [&](int c0, float* v) {
        ld_acc(taddr + (uint32_t)c0, v);
        if (two && r.nkb > 1) {
          float t[COLS];
          ld_acc(taddr + (uint32_t)(TILE_X + c0), t);
#pragma unroll
          for (int j = 0; j < COLS; ++j) v[j] += t[j];
        }
      };
      unsigned int* ticket = p.tickets + ((size_t)r.tile * 2 + rank) * kEpiWarps + ew;
      const size_t fix_acc = 32 * (size_t)p.n_act;            // float4s of one CTA's accumulator
      float4* fix = reinterpret_cast<float4*>(p.fix) + et;
      auto at = [&](int who, int c0) { return fix + (((size_t)who * 2 + rank) * HF + hf) * fix_acc + (size_t)(c0 >> 2) * 128; };
      if (p.S > 1) {
        const int base = r.tile * p.S, self = pair - base;
        // 64-column groups of the tile's accumulators belong to the pairs in turn
        auto owner = [&](int c0) { return (hf * 4 + (c0 >> 6)) % p.S; };
        if (live)
          for (int c0 = c_first; c0 < p.n_act; c0 += C_STEP)
            if (owner(c0) != self) {
              float v[COLS];
              read_acc(c0, v);
              put_fix(at(pair, c0), v);
            }
        __threadfence();
        __syncwarp();
        if (lane == 0) atomicAdd(ticket, 1u);
        if (live && !wait_fix(ticket, kFixDone - 1u, (unsigned)p.S, wc, 226)) live = false;
        live = __all_sync(0xffffffffu, live);
        __threadfence();
        if (live)
          for (int c0 = c_first; c0 < p.n_act; c0 += C_STEP)
            if (owner(c0) == self) {
              float v[COLS];
#pragma unroll
              for (int j = 0; j < COLS; ++j) v[j] = 0.f;
              for (int s = 0; s < p.S; ++s) {               // k order
                float4 o[COLS / 4];
                if (s == self) read_acc(c0, reinterpret_cast<float*>(o));
                else get_fix(at(base + s, c0), o);
                add(o, v);
              }
              finish<KIND>(p, v, unit, quarter, lane, row0, c0, pos_s, kv_s);
            }
        __syncwarp();
        if (lane == 0 && (atomicAdd(ticket, kFixDone) >> 8) == (unsigned)p.S - 1u) *ticket = 0u;       // ready for the next launch
      } else if (parts > 1) {
        // a share's first run goes to part 0 of its pair's place in the buffer, its last one to part 1
        auto place = [&](int share) { return share * 2 + (share * p.per / p.num_kb == r.tile ? 0 : 1); };
        unsigned int t = 0;
        if (lane == 0) t = atomicAdd(ticket, 1u);
        t = __shfl_sync(0xffffffffu, t, 0);
        const bool leave = (int)(t & (kFixDone - 1u)) + 1 < parts;
        if (leave) {
          if (live)
            for (int c0 = c_first; c0 < p.n_act; c0 += C_STEP) {
              float v[COLS];
              read_acc(c0, v);
              put_fix(at(place(pair), c0), v);
            }
          __threadfence();
          __syncwarp();
          if (lane == 0) atomicAdd(ticket, kFixDone);
        } else {
          if (!wait_fix(ticket, ~(kFixDone - 1u), (unsigned)(parts - 1) * kFixDone, wc, 228)) live = false;
          live = __all_sync(0xffffffffu, live);
          __threadfence();
          if (live)
            for (int c0 = c_first; c0 < p.n_act; c0 += C_STEP) {
              float v[COLS];
#pragma unroll
              for (int j = 0; j < COLS; ++j) v[j] = 0.f;
              for (int s = first_share; s <= last_share; ++s) {               // k order
                float4 o[COLS / 4];
                if (s == pair) read_acc(c0, reinterpret_cast<float*>(o));
                else get_fix(at(place(s), c0), o);
                add(o, v);
              }
              finish<KIND>(p, v, unit, quarter, lane, row0, c0, pos_s, kv_s);
            }
          __syncwarp();
          if (lane == 0 && live) *ticket = 0u;                      // ready for the next launch
        }
      } else if (live) {
        for (int c0 = c_first; c0 < p.n_act; c0 += C_STEP) {
          float v[COLS];
          read_acc(c0, v);
          finish<KIND>(p, v, unit, quarter, lane, row0, c0, pos_s, kv_s);
        }
      }
      release(acc);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (p.clk && threadIdx.x == 0) atomicMax(p.clk + kGemmClockSlots, globaltimer_ns());
  // Neither CTA leaves (nor frees its tensor memory) before the other is done: copies, commits and arrivals cross
  // between them until then.  The rendezvous keeps a budget of its own, far above that of the other waits, so that a
  // CTA which has given up still finds its partner.
  if (warp == 2) cluster_meet_before_exit(&meet_bar, 2, lane, wc, &meet_flag_s, 225);
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
}

}  // namespace

// Estimated time of a plan in us, launch included.  Fitted to 600 measured plans (129 .. 4096 rows of the 7B and 13B matrices):
// 11.2 TB/s from L2 to all SMs together, 54 bytes a cycle to one; 6.5 TB/s from HBM, as long as 70 pairs take part; MMAs
// of 256 rows and less than 120 columns take no less time than those of 120 (issuing); reading out an accumulator of 128 lanes
// x 256 columns about 1.5 us, and about as long again for each time it goes through the fix-up buffer.  Over 123 measured shapes
// what it picks is 1 % slower than the fastest plan in the mean, 21 % at the worst (2048 x 5120 x 5120).
static double tile_plan_cost(const TilePlan& g, int N, int K) {
  const double kMHz = 1576.0, n = g.n_act;
  const double waves = g.sk_tiles ? (double)g.tiles / kPairs : (double)((g.tiles * g.S + kPairs - 1) / kPairs);
  const double kbs = !g.sk_tiles ? waves * ((g.num_kb + g.S - 1) / g.S) : g.tiles < kPairs ? (double)g.per : waves * g.num_kb;
  const double tensor = kbs * g.hf * (2 * n > 240 ? 2 * n : 240) / kMHz;
  const double sm = kbs * (g.hf * (double)A_BYTES + 64 * n) / (53.5 * kMHz);
  const double l2 = (double)g.tiles * g.num_kb * (g.hf * 2.0 * A_BYTES + 128 * n) / 11.2e6;
  const double hbm = (double)N * K * 2 / 6.5e6 * (g.pairs < 70 ? 70.0 / g.pairs : 1.0);
  double t = tensor > sm ? tensor : sm;
  if (l2 > t) t = l2;
  if (hbm > t) t = hbm;
  if (g.sk_tiles && g.mchunks > 2) t *= 1.12;               // (shares walk k at their own offsets: L2 serves fewer of them)
  const double drain = 1.45 * n / 256;
  t += 13 + (g.hf == 2 || g.chains == 2 ? (waves < 1 ? 1 : waves) * 1.7 * drain : drain);
  if (g.S > 1) t += 1.7 + 0.95 * g.hf * drain * (g.S - 1) / g.S + (g.hf == 2 ? 1.75 * (g.S - 1) : 0.0);
  if (g.fills > 1) {
    const double over = (waves < 1 ? 1 : waves) * g.fills;              // fills taken over, one after the other
    t += (3 + over) * n / 256;
    if (t < 13 + 3.4 * over * n / 256) t = 13 + 3.4 * over * n / 256;
  }
  if (g.sk_tiles) t += 5.8 + drain * (g.tiles < kPairs ? (g.num_kb + g.per - 1) / g.per - 1 : 1);
  return t;
}

// plain: the fp32 product itself is the result.  max_fix: floats of fix-up buffer that the caller has.
TilePlan make_tile_plan(int M, int N, int K, bool plain, size_t max_fix) {
  TilePlan best;
  double best_t = 0;
  const int least_chunks = (M + TILE_X - 1) / TILE_X;
  // (HF = 2 has no room for two chains: from three chunks of rows on)
  for (int hf = 1; hf <= (least_chunks > 2 && !plain ? 2 : 1); ++hf)
    for (int c = least_chunks; c <= least_chunks + least_chunks / 4 + 2; ++c)
      for (int S = 1; S <= 4 * hf; ++S)
        for (int sk = 0; sk <= (S == 1 && hf == 1 ? 1 : 0); ++sk) {      // (two accumulators per share: never the fastest)
          TilePlan g;
          g.hf = hf;
          g.mchunks = c;
          g.n_act = ((M + c - 1) / c + 31) / 32 * 32;
          g.num_kb = (K + BK - 1) / BK;
          g.tiles = (long long)((N + 256 * hf - 1) / (256 * hf)) * c;
          g.S = S;
          g.sk_tiles = g.per = 0;
          g.fix_floats = 0;
          g.pairs = kPairs;
          if (S > 1) {
            if (g.tiles * S > kPairs || g.num_kb < 4 * S) break;
            g.fix_floats = (size_t)g.tiles * S * 2 * hf * 128 * g.n_act;
          }
          if (g.tiles * S < kPairs) g.pairs = (int)g.tiles * S;
          if (sk) {
            const int rem = (int)(g.tiles % kPairs);
            if (!rem) continue;
            g.sk_tiles = g.tiles < kPairs ? rem : kPairs + rem;
            g.per = (g.sk_tiles * g.num_kb + kPairs - 1) / kPairs;
            if (g.tiles < kPairs && g.per < 4) g.per = 4;
            if (g.tiles < kPairs && g.per >= g.num_kb) continue;          // (as good as whole tiles)
            g.pairs = (g.sk_tiles * g.num_kb + g.per - 1) / g.per;
            g.fix_floats = (size_t)g.pairs * 2 * 2 * hf * 128 * g.n_act;
          }
          if (g.fix_floats > max_fix) continue;
          // a chain is no longer than the product cut evenly over all pairs would make it (in pieces of 4 k blocks at least), nor
          // than half a run
          const int run = sk && g.tiles < kPairs ? g.per : (g.num_kb + S - 1) / S;
          const double piece = 0.9 * ((N + 511) / 512) * g.num_kb * least_chunks / kPairs;
          g.fills = !plain ? 1 : (int)ceil(run / (piece < 4 ? 4 : piece));
          if (plain && g.fills < 2 && run >= 8) g.fills = 2;
          g.fill = (run + g.fills - 1) / g.fills;
          g.chains = !plain && hf == 1 && g.tiles * S <= 2 * kPairs ? 2 : 1;
          const double t = tile_plan_cost(g, N, K);
          if (best_t == 0 || t < best_t) {
            best = g;
            best_t = t;
          }
        }
  return best;
}

Chains gemm_tile_chains(int M, int N, int K) {
  const TilePlan g = make_tile_plan(M, N, K, false);
  Chains c;
  for (int t = 0; t < g.tiles; ++t)
    if (t < g.sk_tiles) {
      for (int u = t * g.num_kb; u < (t + 1) * g.num_kb;) {
        const int share = (u / g.per + 1) * g.per, end = share < (t + 1) * g.num_kb ? share : (t + 1) * g.num_kb;
        c.add(end - u, g.chains);
        u = end;
      }
    } else {
      for (int s = 0; s < g.S; ++s) c.add((s + 1) * g.num_kb / g.S - s * g.num_kb / g.S, g.chains);
    }
  return c;
}

size_t gemm_fix_floats() { return (size_t)kPairs * 2 * 2 * 128 * TILE_X; }

template <int KIND, int HF>
static int launch_kind(const CUtensorMap& tmW, const CUtensorMap& tmX, TileParams q, int pairs, cudaStream_t st) {
  // shared memory left beside the kernel's static variables (barriers; KIND 2: positions and cache rows of a chunk)
  constexpr size_t kRing = 227 * 1024 - 1024 - (KIND == 2 ? 3072 : 512);
  const size_t stage = HF * A_BYTES + (size_t)q.n_act * BK;
  q.stages = (int)(kRing / stage);
  if (q.stages > MAX_STAGES) q.stages = MAX_STAGES;
  static std::atomic<bool> configured{false};
  if (!configured) {
    CERB_CUDA_OK(cudaFuncSetAttribute(gemm_tile_kernel<KIND, HF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kRing + 1024)));
    configured = true;
  }
  // (always the same request: more than half of an SM, so that a CTA may own all of its tensor memory)
  return launch_pdl_cluster(gemm_tile_kernel<KIND, HF>, dim3(2 * pairs), dim3(kThreads), kRing + 1024, st, 2u, tmW, tmX, q) == cudaSuccess ? CERB_OK : CERB_E_CUDA;
}

int launch_gemm_tile(cerb_ctx* c, const CUtensorMap* tmW, const ActMaps* tmX, const TilePlan& g, float* out, float* fix, unsigned int* tickets,
                     int M, int N, int32_t* status, cudaStream_t st, const GemmEpilogue* epi, unsigned long long* clock_slot) {
  const int kind = epi ? epi->kind : 0;
  if (g.tiles * g.num_kb >= (1ll << 30)) return CERB_E_SHAPE;
  if (g.fix_floats && (!fix || !tickets)) return CERB_E_ARG;
  static_assert(2 * kPairs * 2 * kEpiWarps <= kGemmTickets, "one counter per epilogue warp of every split tile");
  TileParams q;
  memset(&q, 0, sizeof(q));
  q.out = kind == 3 ? epi->x : out;
  q.fix = fix; q.tickets = tickets; q.status = status;
  q.M = M; q.N = N;
  q.n_act = g.n_act; q.mchunks = g.mchunks; q.num_kb = g.num_kb; q.tiles = (int)g.tiles;
  q.chains = g.chains; q.fill = g.fill; q.S = g.S; q.sk_tiles = g.sk_tiles; q.per = g.per; q.sk_total = g.sk_tiles * g.num_kb;
  q.wait_cycles = wait_cycles();
  q.clk = clock_slot;
  const CUtensorMap& x = tmX->box(g.n_act / 2);                      // each CTA loads half of a chunk's rows
  if (kind == 1) {
    q.F = N / 2;
    q.act = (bf16*)epi->act;
  }
  if (kind == 2) q.re = *epi->rope;
  auto run = [&](auto hf) {
    constexpr int HF = decltype(hf)::value;
    return kind == 1   ? launch_kind<1, HF>(*tmW, x, q, g.pairs, st)
           : kind == 2 ? launch_kind<2, HF>(*tmW, x, q, g.pairs, st)
           : kind == 3 ? launch_kind<3, HF>(*tmW, x, q, g.pairs, st)
                       : launch_kind<0, 1>(*tmW, x, q, g.pairs, st);
  };
  if (g.hf == 2 && kind == 0) return CERB_E_ARG;
  const int rc = g.hf == 2 ? run(std::integral_constant<int, 2>()) : run(std::integral_constant<int, 1>());
  if (rc != CERB_OK) return rc;
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

}  // namespace cerb
