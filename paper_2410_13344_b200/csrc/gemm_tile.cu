// bf16 GEMM for more than 128 activation rows (batched trees, prefill): output tiles on CTA pairs (tcgen05 cta_group::2).
//
//   D[256 weight rows][up to 256 activation rows] per tile, fp32, in the tensor memory of two CTAs
//
// What bounds it: the tensor pipe from about 512 rows on, weight stream and tensor pipe alike at 256 rows.
//
// Tile.  One MMA is 256 weight rows tall, 128 from each CTA's shared memory, and its activation rows (the MMA's N, up to
// 256) come half from each CTA; each CTA's tensor memory receives its 128 rows of D.  An accumulator takes 256 of the 512
// columns, so there are two, and a tile's epilogue runs under the next tile's MMAs.  A stage is 64 k: 16 KB of weights and
// up to 16 KB of activations per CTA, six or seven stages at 256 rows.  M rows are cut into ceil(M / 256) equal chunks,
// rounded up to 32 rows: 300 rows are two passes of 160, not of 256.
//
// Schedule.  Whole tiles where there are at least as many as pairs: they are dealt out in turn (neighbouring pairs work on
// the chunks of one weight tile, so HBM delivers it once), and what does not fill a last wave evenly, between one and two
// tiles per pair, is cut along k into equal shares, which are done first.  A share is at least one tile long, so at most two
// pairs meet in a tile: the one that finishes first leaves its sums in a fix-up buffer, the other adds them to its own and
// runs the epilogue.  The result has one slot (and the same bits whoever is first).
// Fewer tiles than pairs (a 4096-column GEMM below 1200 rows): the (tile, k block) list is cut into equal shares for all
// pairs and every share leaves its sums in a partial slot of its own, as in gemm_bf16.cu; the kernel that consumes them
// adds the slots.  (A fix-up by one pair would read up to five partial tiles of 256 KB through one SM.)
//
// Epilogues (KIND; only with one slot):
//   1  SwiGLU.  The weight tile is fetched with 16 gate rows and the 16 up rows of the same features in turn (a 4-D view
//      of the matrix), so a warp's 32 accumulator lanes hold 16 (gate, up) pairs; one shuffle per two columns brings the
//      members of a pair together, and half a warp finishes one activation row, the other half the next.
//   2  RoPE and cache append (head_dim 128).  A CTA's 128 weight rows are one head of q, k or v, fetched so that elements i
//      and i + 64 of a rotation pair sit 16 lanes apart (a 5-D view).  Arithmetic and order as in rope_append_kernel.
//   3  Residual add: the tile is added to the fp32 residual stream.
// They replace passes of element-wise kernels over the fp32 sums.
#include <string.h>

#include "tc_common.cuh"

namespace cerb {

namespace {

constexpr int BK = 64;
constexpr int MAX_STAGES = 8;
constexpr int TILE_W = 256;                                // weight rows of a tile (128 per CTA)
constexpr int TILE_X = kGemmRowsPerPass;                   // activation rows of a tile at most
constexpr uint32_t A_BYTES = 128 * BK * 2;
constexpr int kPairs = 74;
constexpr int kEpiWarps = 8;                               // two per 32 tensor-memory lanes, taking 32-column blocks in turn
constexpr int kThreads = 64 + 32 * kEpiWarps;

struct TileParams {
  float* out;               // KIND 0: [slot][M][N]; KIND 3: the residual stream [M][N]
  float* fix;               // [pair][tail, head of a split tile][CTA][column / 4][128 lanes][4]
  unsigned int* tickets;    // [split tile][CTA][epilogue warp], zero on entry and on exit
  bf16* act;                // KIND 1: [M][F]
  RopeEpilogue re;          // KIND 2
  int32_t* status;
  int M, N, F;
  int n_act;                // activation rows per chunk
  int stages;
  int mchunks, num_kb, tiles;
  int sk_tiles, per, sk_total;   // tiles cut along k, k blocks per share, k blocks in all of them
  int nslots;
  long long wait_cycles;
  unsigned long long* clk;
};

// A run of k blocks inside one tile.
struct Run {
  int tile, kb0, nkb;
};
struct Work {
  int u, u1, whole, step, tiles, num_kb;
  __device__ __forceinline__ Work(const TileParams& p, int pair, int pairs)
      : u(pair * p.per), u1(min(pair * p.per + p.per, p.sk_total)), whole(p.sk_tiles + pair), step(pairs), tiles(p.tiles), num_kb(p.num_kb) {}
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
    r.kb0 = 0;
    r.nkb = num_kb;
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

// Finishes 32 columns (activation rows row0 + c0 ...) of one accumulator lane.  Everything is computed before anything is
// stored: with the bounds checks of the stores in between, each column's chain of latencies came after the last one's
// (QKV of the 7B shape at 512 rows: 103 us, and 58 this way with eight epilogue warps instead of four).
template <int KIND>
__device__ __forceinline__ void finish(const TileParams& p, const float* v, int slot, int unit, int quarter, int lane, int row0, int c0,
                                       const int* pos_s, const int* kv_s) {
  const int left = min(32, min(p.n_act - c0, p.M - row0 - c0));            // live columns
  if constexpr (KIND == 0 || KIND == 3) {
    const int n_out = unit * 128 + quarter * 32 + lane;
    if (n_out >= p.N) return;
    float* o = p.out + ((size_t)slot * p.M + row0 + c0) * p.N + n_out;     // (consecutive lanes: consecutive columns of a row)
    float x[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) x[j] = KIND == 3 && j < left ? o[(size_t)j * p.N] : 0.f;
    if (left == 32) {
#pragma unroll
      for (int j = 0; j < 32; ++j) o[(size_t)j * p.N] = KIND == 3 ? x[j] + v[j] : v[j];
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (j < left) o[(size_t)j * p.N] = KIND == 3 ? x[j] + v[j] : v[j];
    }
  } else {
    const int hi = lane >> 4;
    const int i = quarter * 16 + (lane & 15);                               // feature / rotation index inside the unit
    // lanes 0-15 hold the first member of each pair (gate; element i), lanes 16-31 the second (up; element i + 64):
    // the lower half of the warp finishes column 2 j, the upper half column 2 j + 1
    float a[16], b[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const float got = __shfl_xor_sync(0xffffffffu, hi ? v[2 * j] : v[2 * j + 1], 16);
      a[j] = hi ? got : v[2 * j];
      b[j] = hi ? v[2 * j + 1] : got;
    }
    if constexpr (KIND == 1) {
      const int f = unit * 64 + i;
#pragma unroll
      for (int j = 0; j < 16; ++j) a[j] = a[j] / (1.0f + expf(-a[j])) * b[j];
      if (f >= p.F) return;
      bf16* o = p.act + (size_t)(row0 + c0 + hi) * p.F + f;
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (2 * j + hi < left) o[(size_t)(2 * j) * p.F] = __float2bfloat16_rn(a[j]);
    } else {
      if (unit >= 3 * p.re.H) return;
      const int which = unit / p.re.H, h = unit - which * p.re.H;
      int kv[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) kv[j] = 2 * j + hi < left ? kv_s[c0 + 2 * j + hi] : -1;
      if (which < 2) {
        float2 cs[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int pos = pos_s[c0 + 2 * j + hi];
          cs[j] = p.re.rope[(size_t)(pos < 0 ? 0 : pos) * 64 + i];
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float o1 = a[j] * cs[j].x - b[j] * cs[j].y;
          b[j] = b[j] * cs[j].x + a[j] * cs[j].y;
          a[j] = o1;
        }
      }
      bf16* q = reinterpret_cast<bf16*>(p.re.q) + ((size_t)(row0 + c0 + hi) * p.re.H + h) * 128 + i;
      bf16* pool = reinterpret_cast<bf16*>(which == 1 ? p.re.kpool : p.re.vpool) + (size_t)h * CERB_PAGE * 128 + i;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        bf16* o = which == 0 ? q + (size_t)(2 * j) * p.re.H * 128 : pool + (size_t)kv[j] * 128;
        if (kv[j] >= 0) {
          o[0] = __float2bfloat16_rn(a[j]);
          o[64] = __float2bfloat16_rn(b[j]);
        }
      }
    }
  }
}

// A share's half of a split tile, warp by warp: whichever of the two pairs comes first (a ticket) leaves its sums in the
// fix-up buffer and says so; the other one waits for that (the first has finished its MMAs, so nothing but its stores is
// waited for) and adds them to its own, which have stayed in tensor memory.
constexpr unsigned int kFixDone = 16u;
__device__ __forceinline__ bool wait_fix(const unsigned int* ticket, const WaitCtx& w, int site) {
  const long long t0 = clock64();
  const long long budget = *w.aborted ? kAbortedWaitCycles : w.budget;
  for (;;) {
    for (int i = 0; i < 16; ++i) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ticket) : "memory");
      if (v & kFixDone) return true;
    }
    if (clock64() - t0 > budget) break;
  }
  wait_ran_out(w, site);
  return false;
}

template <int KIND>
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
  const uint32_t stage_bytes = A_BYTES + (uint32_t)p.n_act * BK;               // (half the chunk's activation rows)
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
      mbar_init(smem_u32(&acc_empty[i]), 2 * kEpiWarps);
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
        load_weights<KIND>(smem_base + (uint32_t)qw.s * stage_bytes, &tmW, rw.kb0, (rw.tile / p.mchunks) * 2 + rank,
                           mapa_u32(smem_u32(&full_bar[qw.s]), 0), pol_w);
        ++rw.kb0;
        --rw.nkb;
        qw.next(p.stages);
      };
      auto load_x = [&]() {
        if (rx.nkb == 0) wx.next(rx);
        tma_load_2d_pair(smem_base + (uint32_t)qx.s * stage_bytes + A_BYTES, &tmX, rx.kb0 * BK, (rx.tile % p.mchunks) * p.n_act + rank * (p.n_act >> 1),
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
      const uint32_t idesc = idesc_bf16(TILE_W, (uint32_t)p.n_act, false, false);
      Work w(p, pair, pairs);
      Run r;
      Ring q;
      bool live = true;
      for (int g = 0; live && w.next(r); ++g) {
        const int buf = g & 1;
        if (!mbar_wait_cluster(smem_u32(&acc_empty[buf]), ((uint32_t)(g >> 1) & 1u) ^ 1u, wc, 222)) live = false;
        live = __all_sync(0xffffffffu, live);
        tc_fence_after();
        const uint32_t d = tmem_base + (uint32_t)(buf * TILE_X);
        for (int k = 0; live && k < r.nkb; ++k) {
          if (!mbar_wait_cluster(smem_u32(&full_bar[q.s]), q.ph, wc, 223)) live = false;
          live = __all_sync(0xffffffffu, live);
          if (!live) break;
          tc_fence_after();
          const uint32_t src = smem_base + (uint32_t)q.s * stage_bytes;
          const uint64_t adesc = desc_k_sw128(src), bdesc = desc_k_sw128(src + A_BYTES);
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
              umma_bf16_pair(d, adesc + (uint64_t)(kk * 2), bdesc + (uint64_t)(kk * 2), idesc, (k > 0 || kk > 0) ? 1u : 0u);
            umma_commit_pair(smem_u32(&empty_bar[q.s]));       // the stage is free in both CTAs once these MMAs have read it
            if (k + 1 == r.nkb) umma_commit_pair(smem_u32(&acc_full[buf]));
          }
          __syncwarp();
          q.next(p.stages);
        }
      }
      if (!live && elect_one()) {
        asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&drain_bar)) : "memory");
        mbar_wait_drain(smem_u32(&drain_bar), 0, 40000000ll);
      }
    }
  } else {
    const int quarter = warp & 3;                    // tensor-memory lanes 32 * quarter .. + 31 belong to this warp
    const int ew = warp - 2, half = ew >> 2;         // columns: 32-column blocks half, half + 2, ...
    const int et = quarter * 32 + lane;
    griddep_wait();                                  // the kernels before this one may still be reading what this one writes
    const uint32_t ae[2] = {mapa_u32(smem_u32(&acc_empty[0]), 0), mapa_u32(smem_u32(&acc_empty[1]), 0)};
    Work w(p, pair, pairs);
    Run r;
    int chunk_known = -1;
    // A warp whose wait has run out writes nothing more, but goes through the remaining runs (every later wait is short
    // then): the other epilogue warps meet it at named barriers.
    bool live = true;
    for (int g = 0; w.next(r); ++g) {
      const int buf = g & 1;
      const int tile_w = r.tile / p.mchunks, chunk = r.tile % p.mchunks;
      const int unit = tile_w * 2 + rank, row0 = chunk * p.n_act;
      if (KIND == 2 && chunk != chunk_known) {
        // positions and cache rows of the chunk's activation rows
        asm volatile("bar.sync 2, 256;" ::: "memory");                       // (the previous tile's readers are done)
        const RopeEpilogue& e = p.re;
        for (int c = ew * 32 + lane; c < p.n_act; c += 32 * kEpiWarps) {
          int pos = -1, kv = -1;
          if (row0 + c < p.M) {
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
        asm volatile("bar.sync 2, 256;" ::: "memory");
        chunk_known = chunk;
      }
      if (!mbar_wait_cluster(smem_u32(&acc_full[buf]), (uint32_t)(g >> 1) & 1u, wc, 224)) live = false;      // the output is undefined from here on
      live = __all_sync(0xffffffffu, live);
      tc_fence_after();
      const uint32_t taddr = tmem_base + (uint32_t)(buf * TILE_X) + ((uint32_t)(quarter * 32) << 16);
      int first_share = pair, last_share = pair;
      if (r.tile < p.sk_tiles) {
        first_share = r.tile * p.num_kb / p.per;
        last_share = (r.tile * p.num_kb + p.num_kb - 1) / p.per;
      }
      const bool split = p.nslots == 1 && last_share > first_share;         // (two pairs: the first has the tile's head)
      // fix-up buffer: a pair has at most one tail (part 0) and one head (part 1) of a split tile
      const size_t fix_tile = (size_t)128 * p.n_act;
      const bool head = pair == first_share;
      float4* mine = reinterpret_cast<float4*>(p.fix + ((size_t)(pair * 2 + (head ? 1 : 0)) * 2 + rank) * fix_tile) + et;
      const float4* other = reinterpret_cast<const float4*>(p.fix + ((size_t)(head ? last_share * 2 : first_share * 2 + 1) * 2 + rank) * fix_tile) + et;
      unsigned int* ticket = p.tickets + ((size_t)r.tile * 2 + rank) * kEpiWarps + ew;
      bool leave = false;
      if (split) {
        unsigned int t = 0;
        if (lane == 0) t = atomicAdd(ticket, 1u);
        t = __shfl_sync(0xffffffffu, t, 0);
        leave = t == 0u;
        if (!leave && !(t & kFixDone)) {
          if (!wait_fix(ticket, wc, 226)) live = false;
          live = __all_sync(0xffffffffu, live);
        }
        if (!leave) __threadfence();
      }
      if (live)
        for (int c0 = half * 32; c0 < p.n_act; c0 += 64) {
          float v[32];
          float4 o4[8];
          if (split && !leave) {
#pragma unroll
            for (int j = 0; j < 8; ++j) o4[j] = __ldcg(other + (size_t)((c0 >> 2) + j) * 128);
          }
          tmem_ld16_nowait(taddr + (uint32_t)c0, reinterpret_cast<uint32_t*>(v));
          tmem_ld16_nowait(taddr + (uint32_t)c0 + 16u, reinterpret_cast<uint32_t*>(v + 16));
          tmem_ld_wait();
          if (leave) {
#pragma unroll
            for (int j = 0; j < 8; ++j) __stcg(mine + (size_t)((c0 >> 2) + j) * 128, make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]));
          } else {
            if (split) {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                v[4 * j] += o4[j].x; v[4 * j + 1] += o4[j].y; v[4 * j + 2] += o4[j].z; v[4 * j + 3] += o4[j].w;
              }
            }
            finish<KIND>(p, v, p.nslots > 1 ? pair - first_share : 0, unit, quarter, lane, row0, c0, pos_s, kv_s);
          }
        }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(ae[buf]);          // (the first CTA's own warps arrive the same way)
      if (split) {
        __threadfence();
        __syncwarp();
        if (lane == 0) {
          if (leave) atomicAdd(ticket, kFixDone);
          else if (live) *ticket = 0u;                      // ready for the next launch
        }
      }
      if (KIND == 0 && p.nslots > 1 && pair == last_share) {
        // slots this tile does not use
        const int n_out = unit * 128 + et;
        const int rows = min(p.n_act, p.M - row0);
        if (half == 0 && n_out < p.N)
          for (int z = last_share - first_share + 1; z < p.nslots; ++z) {
            float* zo = p.out + ((size_t)z * p.M + row0) * p.N + n_out;
            for (int m = 0; m < rows; ++m) { *zo = 0.f; zo += p.N; }
          }
      }
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

// max_slots, max_fix: what the caller's scratch holds (partial slots per output, floats of fix-up buffer).
TilePlan make_tile_plan(int M, int N, int K, int max_slots, size_t max_fix) {
  TilePlan g;
  g.mchunks = (M + TILE_X - 1) / TILE_X;
  g.n_act = ((M + g.mchunks - 1) / g.mchunks + 31) / 32 * 32;
  g.num_kb = (K + BK - 1) / BK;
  g.tiles = (long long)((N + TILE_W - 1) / TILE_W) * g.mchunks;
  g.whole = g.tiles >= kPairs;
  g.pairs = kPairs;
  g.nslots = 1;
  g.sk_tiles = 0;
  g.per = 0;
  g.fix_floats = 0;
  if (g.whole) {
    const int rem = (int)(g.tiles % kPairs);
    const size_t fix = (size_t)kPairs * 2 * 2 * 128 * g.n_act;
    if (rem && fix <= max_fix) {
      g.sk_tiles = kPairs + rem;
      g.per = (g.sk_tiles * g.num_kb + kPairs - 1) / kPairs;
      g.fix_floats = fix;
    }
    return g;
  }
  g.sk_tiles = (int)g.tiles;
  const int total = g.sk_tiles * g.num_kb;
  g.per = (total + kPairs - 1) / kPairs;
  const int least = g.num_kb < 4 ? g.num_kb : 4;      // do not shred tiny problems into one-block shares
  if (g.per < least) g.per = least;
  for (;; ++g.per) {
    g.nslots = 1;
    for (int t = 0; t < g.sk_tiles; ++t) {
      const int n = (t * g.num_kb + g.num_kb - 1) / g.per - t * g.num_kb / g.per + 1;
      if (n > g.nslots) g.nslots = n;
    }
    if (g.nslots <= max_slots) break;                  // (a share of num_kb blocks leaves one slot)
  }
  g.pairs = (total + g.per - 1) / g.per;
  return g;
}

size_t gemm_fix_floats() { return (size_t)kPairs * 2 * 2 * 128 * TILE_X; }

template <int KIND>
static int launch_kind(const CUtensorMap& tmW, const CUtensorMap& tmX, TileParams q, int pairs, cudaStream_t st) {
  // shared memory left beside the kernel's static variables (barriers; KIND 2: positions and cache rows of a chunk)
  constexpr size_t kRing = 227 * 1024 - 1024 - (KIND == 2 ? 3072 : 512);
  const size_t stage = A_BYTES + (size_t)q.n_act * BK;
  q.stages = (int)(kRing / stage);
  if (q.stages > MAX_STAGES) q.stages = MAX_STAGES;
  static bool configured = false;
  if (!configured) {
    CERB_CUDA_OK(cudaFuncSetAttribute(gemm_tile_kernel<KIND>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kRing + 1024)));
    configured = true;
  }
  // (always the same request: more than half of an SM, so that a CTA may own all of its tensor memory)
  return launch_pdl_cluster(gemm_tile_kernel<KIND>, dim3(2 * pairs), dim3(kThreads), kRing + 1024, st, 2u, tmW, tmX, q) == cudaSuccess ? CERB_OK : CERB_E_CUDA;
}

int launch_gemm_tile(cerb_ctx* c, const CUtensorMap* tmW, const ActMaps* tmX, const TilePlan& g, float* out, float* fix, unsigned int* tickets,
                     int M, int N, int32_t* status, cudaStream_t st, const GemmEpilogue* epi, unsigned long long* clock_slot) {
  const int kind = epi ? epi->kind : 0;
  if (g.tiles >= (1ll << 30) || (long long)g.sk_tiles * g.num_kb >= (1ll << 30)) return CERB_E_SHAPE;
  if (kind != 0 && !g.whole) return CERB_E_SHAPE;
  if (g.whole && g.sk_tiles && (!fix || !tickets)) return CERB_E_ARG;
  static_assert(2 * kPairs * 2 * kEpiWarps <= kGemmTickets, "one ticket per epilogue warp of every split tile");
  TileParams q;
  memset(&q, 0, sizeof(q));
  q.out = kind == 3 ? epi->x : out;
  q.fix = fix; q.tickets = tickets; q.status = status;
  q.M = M; q.N = N;
  q.n_act = g.n_act; q.mchunks = g.mchunks; q.num_kb = g.num_kb; q.tiles = (int)g.tiles;
  q.sk_tiles = g.sk_tiles; q.per = g.per; q.sk_total = g.sk_tiles * g.num_kb; q.nslots = g.nslots;
  q.wait_cycles = wait_cycles();
  q.clk = clock_slot;
  const CUtensorMap& x = tmX->box(g.n_act / 2);                      // each CTA loads half of a chunk's rows
  int rc;
  if (kind == 1) {
    q.F = N / 2;
    q.act = (bf16*)epi->act;
    rc = launch_kind<1>(*tmW, x, q, g.pairs, st);
  } else if (kind == 2) {
    q.re = *epi->rope;
    rc = launch_kind<2>(*tmW, x, q, g.pairs, st);
  } else if (kind == 3) {
    rc = launch_kind<3>(*tmW, x, q, g.pairs, st);
  } else {
    rc = launch_kind<0>(*tmW, x, q, g.pairs, st);
  }
  if (rc != CERB_OK) return rc;
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

}  // namespace cerb
