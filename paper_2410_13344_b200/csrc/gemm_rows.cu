// bf16 GEMM of 9 to 256 activation rows in tiles as wide as an SM's share: gate-up with SwiGLU, QKV with RoPE and cache append, whose outputs are
// finished where they are summed, and plain sums (O, down, up to 128 rows the LM head) in few parts of k.
//
//   CG = 1:  D[128 activation rows][w weight rows] per CTA
//   CG = 2:  D[256 activation rows][2 w weight rows] per pair of CTAs (cta_group::2), fp32, in tensor memory; one tile each, of all of k or of a part of it
//
// What bounds it: the weight stream up to 64 rows, then L2 on its way to the SMs.  The activation rows are the MMA's M side (rows that do not exist
// are whatever lies behind them in shared memory; they only reach accumulator rows that nobody reads), the weight rows its N side, which comes
// in steps of 16: so a matrix is cut into as many equal tiles as there are SMs, every output has one sum in one place, and no partial
// sums, no exchange and no kernel behind the product are needed.  (Weights on the M side come in steps of 128 or 256 rows: 86 tiles of a
// 22016-row matrix for 148 SMs or 74 pairs had to be cut along k.)
//
// Weight tile of a CTA.  Groups of eight rows, one 8 x 128-byte swizzle atom each:
//   SwiGLU: the gate rows of four neighbouring features, then their up rows (4-D view of the matrix);
//   plain sums: neighbouring rows;
//   RoPE (head_dim 128): elements i .. i + 3 of a head, then i + 64 .. i + 67; a tile has the same four rotations of `groups` heads, so that a
//   thread (one activation row) keeps its angles in registers (4-D view; 16 tiles per block of heads).
// An epilogue thread thus finds both members of every pair among its own columns.
// A pair's MMA takes half of the activation rows and half of the weight rows from each CTA: each CTA's accumulator has its half of the
// rows and the columns of both.  That halves the activations that each SM fetches.
//
// Issuers and chains.  One thread waits for a stage, issues four MMAs and commits them in 600 to 670 cycles, whatever the MMAs' size up to 160 columns
// (80 cycles each are possible); it issues nothing while it waits, and two accumulators of its own change nothing.  Two warps that take the
// stages in turn need 320 to 340 per stage, three 225.  Each has one accumulator or several in turn: the tensor cores cut a running sum off towards
// zero at every step, so a sum is made of several short chains, as many as it takes for them to be no longer than those of the kernel that the
// product goes to otherwise (plan_ring; where they do not fit, it goes there).  V of a first layer against float64, by the bf16 values that round the
// other way, in 1e-6 of their size, 32 / 128 rows: 2048 columns 0.48 / 0.26 there, 0.75 / 0.39 in three / four chains, 0.27 / 0.30 in six; 2560 columns 0.37 / 0.56,
// 0.62 / 0.93 in three, 0.29 / 0.39 in six; 4096 columns, 96 rows 1.23, 1.41 in three, 1.09 in four.  Six chains instead of four cost 0.2 us a launch.
// A pair's tile of more than 256 columns is three MMAs wide: two of 96 columns each, whose accumulators go over to a third one of that size in turn, while
// the epilogue warps add what the last one holds to their registers (which have room for these 192 columns, and for no more), and one of the
// rest, with an accumulator for either half of k; two warps issue the two kinds.  (7B width: chains of 8 and 16 k blocks and of 32, 23 in the root mean square, 24 in cut output
// tiles; activations of 160 / 256 rows 4.4 / 5.0e-6 from float64 as above, 4.8 / 5.7e-6 there.  Two MMAs with one change each, chains of 30 and 34: 6.7 / 7.5e-6,
// and 0.5 % less for a forward: 1287 / 1297 us of 256 rows, 8 layers.)
//
// Roles (512 threads): warp 0 = TMA producer (one lane), which fills the ring with weights ahead of the dependency wait; warps 1 to 3 = MMA
// issuers (of a pair's first CTA); warps 4 to 15 = epilogue, three per 32 accumulator rows.
#include <string.h>

#include <type_traits>

#include "tc_common.cuh"

namespace cerb {

namespace {

constexpr int BK = 64;
constexpr int MAX_STAGES = 18;
constexpr int ROWS = 128;                                  // accumulator rows of a CTA
constexpr int kSms = 148;
constexpr int kIssuers = 3;                                // at most
constexpr int kParts = 3;                                  // epilogue warps per 32 accumulator rows
constexpr int kThreads = 128 + 128 * kParts;
constexpr int COLS = 16;                                   // columns an epilogue warp takes at a time (two groups)
constexpr int HELD = 2;                                    // blocks of columns of each of two MMAs that an epilogue thread holds
constexpr int kTurnCols = HELD * kParts * COLS;            // columns of such an MMA
constexpr int kTurnGroups = kTurnCols / 16;                // groups of either CTA in it
constexpr size_t kRing = 226 * 1024;                       // shared memory of the ring, with what the last stage's missing rows need

struct RowsParams {
  float* out;               // KIND 0: [part][M][N]
  int N, parts;             // KIND 0: columns of the output, pieces that k is cut into
  bf16* act;                // KIND 1: [M][F]
  RopeEpilogue re;          // KIND 2
  int32_t* status;
  int M, F, num_kb;
  int groups;               // groups of eight weight rows of a CTA
  int x_rows;               // activation rows fetched by a CTA
  int m_rows;               // rows of a CTA's accumulator: 128, or (CG = 1) 64, of which each warp quarter has 16
  int stages, issuers, chains;
  int turn, turns;          // three MMAs: k blocks from one change of accumulators to the next, and how many of these there are; else 0
  uint32_t acc_cols, tmem_cols;
  long long wait_cycles;
  unsigned long long* clk;
};

template <int CG>
__device__ __forceinline__ void load_groups(uint32_t dst, const CUtensorMap* map, int x, int row, int group, uint32_t bar, uint64_t pol) {
  if constexpr (CG == 1)
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
        ::"r"(dst), "l"((uint64_t)map), "r"(x), "r"(row), "r"(0), "r"(group), "r"(bar), "l"(pol)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
        ::"r"(dst), "l"((uint64_t)map), "r"(x), "r"(row), "r"(0), "r"(group), "r"(bar), "l"(pol)
        : "memory");
}

// MANY: more than four accumulators.  (An instance of its own: with the loop for them in the others, where it does not run, 8 layers of 4096 columns took 774 instead of
// 768 us at 9 rows.)
template <int KIND, int CG, bool MANY>
__global__ void __launch_bounds__(kThreads, 1) gemm_rows_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                                                                const RowsParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[MAX_STAGES];      // CG = 2: used in the pair's first CTA only
  __shared__ __align__(8) uint64_t empty_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t acc_full, drain_bar[kIssuers];
  __shared__ __align__(8) uint64_t turn_full, turn_done, meet_bar;       // turn_done: first CTA only, all epilogue warps of the pair arrive
  __shared__ uint32_t tmem_base_slot;
  __shared__ int aborted_s, meet_flag_s;
  volatile int* aborted = &aborted_s;
  const WaitCtx wc{p.wait_cycles, aborted, p.status, KIND + 10 * p.num_kb + 100000 * p.M};

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t w_bytes = (uint32_t)p.groups * 1024u;
  const uint32_t stage_bytes = w_bytes + (uint32_t)p.x_rows * 128u;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;       // (one value per warp, as the compiler sees)
  const int rank = CG == 2 ? (int)cluster_ctarank() : 0;
  const bool first = rank == 0;
  const bool turning = KIND == 1 && CG == 2 && p.turns > 0;                // three MMAs per 16 k
  // Consecutive groups; RoPE: four rotations of a block of heads.  Plain sums: the parts of a tile are neighbours.
  const int row0 = KIND == 2 ? ((int)blockIdx.x & 15) * 4 : 0;
  const int tile = KIND == 2 ? (int)blockIdx.x >> 4 : KIND == 0 ? (int)blockIdx.x / CG / p.parts : (int)blockIdx.x;
  const int slot = KIND == 0 ? (int)blockIdx.x / CG - tile * p.parts : 0;
  const int group0 = (KIND == 0 ? tile * CG + rank : tile) * p.groups;
  const int kb0 = KIND == 0 ? slot * p.num_kb / p.parts : 0, num_kb = KIND == 0 ? (slot + 1) * p.num_kb / p.parts - kb0 : p.num_kb;

  if (threadIdx.x == 0) {
    aborted_s = 0;
    meet_flag_s = 0;
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), turning ? 2 : 1);
    }
    mbar_init(smem_u32(&acc_full), (uint32_t)p.issuers);
    for (int i = 0; i < kIssuers; ++i) mbar_init(smem_u32(&drain_bar[i]), 1);
    if constexpr (CG == 2) {
      mbar_init(smem_u32(&turn_full), 1);
      mbar_init(smem_u32(&turn_done), 2 * 4 * kParts);
      mbar_init(smem_u32(&meet_bar), 2);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if constexpr (CG == 1) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(p.tmem_cols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    } else {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(p.tmem_cols) : "memory");
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if constexpr (CG == 2) {
    cluster_start_arrive();       // the other CTA's barriers exist before anything is signalled across
    cluster_start_wait();
  }
  const uint32_t tmem_base = tmem_base_slot;
  auto wait = [&](uint64_t& bar, uint32_t parity, int site) {
    return CG == 2 ? mbar_wait_cluster(smem_u32(&bar), parity, wc, site) : mbar_wait(smem_u32(&bar), parity, wc, site);
  };

  if (warp == 0) {
    if (lane == 0) {
      const uint64_t pol_w = l2_policy(true), pol_x = l2_policy(false);
      auto full = [&](int s) { return CG == 2 ? mapa_u32(smem_u32(&full_bar[s]), 0) : smem_u32(&full_bar[s]); };
      auto load_w = [&](int kb, int s) {
        if (first) mbar_expect_tx(smem_u32(&full_bar[s]), CG * stage_bytes);               // (a pair's first CTA counts both CTAs' copies)
        if constexpr (KIND == 0 && CG == 2) tma_load_2d_pair(smem_base + (uint32_t)s * stage_bytes, &tmW, (kb0 + kb) * BK, group0 * 8, full(s), pol_w);
        else if constexpr (KIND == 0) tma_load_2d_hint(smem_base + (uint32_t)s * stage_bytes, &tmW, (kb0 + kb) * BK, group0 * 8, full(s), pol_w);
        else load_groups<CG>(smem_base + (uint32_t)s * stage_bytes, &tmW, kb * BK, row0, group0, full(s), pol_w);
      };
      auto load_x = [&](int kb, int s) {
        const uint32_t dst = smem_base + (uint32_t)s * stage_bytes + w_bytes;
        if constexpr (CG == 2) tma_load_2d_pair(dst, &tmX, (kb0 + kb) * BK, rank * p.x_rows, full(s), pol_x);
        else tma_load_2d_hint(dst, &tmX, (kb0 + kb) * BK, 0, full(s), pol_x);
      };
      const int pre = min(num_kb, p.stages);
      for (int i = 0; i < pre; ++i) load_w(i, i);
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmX) : "memory");
      griddep_wait();
      griddep_launch();                                    // (only now: see launch_order.cu)
      if (p.clk) atomicMin(p.clk, globaltimer_ns());
      for (int i = 0; i < pre; ++i) load_x(i, i);
      int issued = pre, s = 0;
      uint32_t ph = 0;
      for (int i = pre; i < num_kb; ++i) {
        if (!wait(empty_bar[s], ph, 241)) break;
        load_w(i, s);
        load_x(i, s);
        issued = i + 1;
        if (++s == p.stages) { s = 0; ph ^= 1u; }
      }
      if (*aborted) {
        // give-up path: the copies already issued still land in this CTA's shared memory; see each of them in.  (A pair's are counted on
        // the first CTA's barriers, and the CTAs may have stopped at different stages: both let the time of many round trips pass, too.)
        if (first)
          for (int i = issued > p.stages ? issued - p.stages : 0; i < issued; ++i)
            mbar_wait_drain(smem_u32(&full_bar[i % p.stages]), (uint32_t)(i / p.stages) & 1u, CG == 2 ? 2000000ll : kDrainCycles);
        const long long t_land = clock64();
        while (CG == 2 && clock64() - t_land < 400000ll) __nanosleep(1000);
      }
    }
  } else if (warp <= kIssuers) {
    const int self = warp - 1;
    if (first && self < p.issuers) {
      bool live = true;
      auto commit = [&](uint64_t& bar) {
        if constexpr (CG == 2) umma_commit_pair(smem_u32(&bar));
        else umma_commit(smem_u32(&bar));
      };
      auto issue = [&](int s, int groups_at, uint32_t idesc, uint32_t d, bool fresh) {
        const uint32_t src = smem_base + (uint32_t)s * stage_bytes;
        const uint64_t adesc = desc_k_sw128(src + w_bytes), bdesc = desc_k_sw128(src + (uint32_t)groups_at * 1024u);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk) {
          const uint32_t acc = (!fresh || kk > 0) ? 1u : 0u;
          if constexpr (CG == 2) umma_bf16_pair(d, adesc + (uint64_t)(kk * 2), bdesc + (uint64_t)(kk * 2), idesc, acc);
          else umma_bf16(d, adesc + (uint64_t)(kk * 2), bdesc + (uint64_t)(kk * 2), idesc, acc);
        }
      };
      if (!turning) {
        const uint32_t idesc = idesc_bf16(CG * (uint32_t)p.m_rows, p.acc_cols, false, false);
        // this issuer's accumulators, which it takes in turn
        const uint32_t d0 = tmem_base + (uint32_t)self * p.acc_cols, d_end = tmem_base + (uint32_t)p.chains * p.acc_cols;
        uint32_t d = d0, ph = 0;
        int s = self;
        for (int i = self; i < num_kb; i += p.issuers) {
          live = __all_sync(0xffffffffu, wait(full_bar[s], ph, 242));
          if (!live) break;
          tc_fence_after();
          if (elect_one()) {
            issue(s, 0, idesc, d, i < p.chains);
            commit(empty_bar[s]);                              // the stage is free once the MMAs have read it
          }
          __syncwarp();
          d += (uint32_t)p.issuers * p.acc_cols;
          if (d >= d_end) d = d0;
          if ((s += p.issuers) >= p.stages) { s = self; ph ^= 1u; }
        }
      } else {
        const uint32_t idesc_t = idesc_bf16(2 * ROWS, kTurnCols, false, false);
        const uint32_t rest = 16u * (uint32_t)p.groups - 2 * kTurnCols, idesc_r = idesc_bf16(2 * ROWS, rest, false, false);
        uint32_t d0 = tmem_base, d1 = d0 + kTurnCols, spare = d1 + kTurnCols, ph = 0;              // the first issuer's
        uint32_t d = tmem_base + 3 * kTurnCols;                                                   // the second one's
        bool fresh0 = true, fresh1 = true;
        int t = 0;                                             // changes so far
        for (int i = 0, s = 0; i < num_kb; ++i) {
          if (self == 1) {
            fresh0 = i == 0 || i == num_kb / 2;
            if (i > 0 && fresh0) d += rest;
          } else if (t < p.turns && i == (t + 1) * p.turn) {
            // the spare accumulator has been taken over since the last change
            live = t == 0 || __all_sync(0xffffffffu, wait(turn_done, (uint32_t)(t - 1) & 1u, 244));
            if (!live) break;
            tc_fence_after();
            if (elect_one()) commit(turn_full);
            __syncwarp();
            uint32_t& mine = t & 1 ? d1 : d0;
            const uint32_t done = mine;
            mine = spare;
            spare = done;
            (t & 1 ? fresh1 : fresh0) = true;
            ++t;
          }
          live = __all_sync(0xffffffffu, wait(full_bar[s], ph, 242));
          if (!live) break;
          tc_fence_after();
          if (elect_one()) {
            if (self == 0) {
              issue(s, 0, idesc_t, d0, fresh0);
              issue(s, kTurnGroups, idesc_t, d1, fresh1);
            } else {
              issue(s, 2 * kTurnGroups, idesc_r, d, fresh0);
            }
            commit(empty_bar[s]);
          }
          __syncwarp();
          fresh0 = fresh1 = false;
          if (++s == p.stages) { s = 0; ph ^= 1u; }
        }
      }
      if (elect_one()) {
        if (live) commit(acc_full);
        if (!live || *aborted) {
          // give-up path, whoever's wait ran out: the MMAs already issued still read shared memory and write tensor memory; see them retire
          if constexpr (CG == 2)
            asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(&drain_bar[self])) : "memory");
          else umma_commit(smem_u32(&drain_bar[self]));
          mbar_wait_drain(smem_u32(&drain_bar[self]), 0, CG == 2 ? 40000000ll : kDrainCycles);
        }
      }
    }
  } else if (warp >= 4) {
    const int quarter = warp & 3, part = (warp >> 2) - 1;
    const int per_quarter = p.m_rows / 4, own = quarter * per_quarter + lane, row = rank * p.x_rows + own;
    griddep_wait();
    bool ok = lane < per_quarter && own < p.x_rows && row < p.M;
    float cs[CG][4], sn[CG][4];
    size_t kv = 0;
    if constexpr (KIND == 2) {
      // where the row's key goes, and its rotations: on the way while the products run
      const RopeEpilogue& e = p.re;
      if (ok) {
        int b, v;
        locate_row(row, e.row_off, e.B, e.n, b, v);
        const int len = e.len[b], pos = len + e.depth[v], slot = len + v;
        ok = v < e.n_active[b] && pos < e.max_pos && slot < e.max_pos;
        if (ok) {
          kv = (size_t)e.page_table[(size_t)b * e.max_pages + slot / CERB_PAGE] * e.H * CERB_PAGE + slot % CERB_PAGE;
#pragma unroll
          for (int r = 0; r < CG; ++r) {
            const float4* rot = reinterpret_cast<const float4*>(e.rope + (size_t)pos * 64 + row0 + (r - rank) * 4);
            const float4 r0 = rot[0], r1 = rot[1];
            cs[r][0] = r0.x; sn[r][0] = r0.y; cs[r][1] = r0.z; sn[r][1] = r0.w;
            cs[r][2] = r1.x; sn[r][2] = r1.y; cs[r][3] = r1.z; sn[r][3] = r1.w;
          }
        }
      }
    }
    const uint32_t lanes = tmem_base + ((uint32_t)(quarter * 32) << 16);
    bool live = rank * p.x_rows + quarter * per_quarter < p.M && quarter * per_quarter < p.x_rows;      // (a warp none of whose rows exist reads no accumulator)
    float held[2][CG == 2 && KIND == 1 ? HELD : 1][COLS];
    uint32_t at0 = lanes, at1 = at0 + kTurnCols, spare = at1 + kTurnCols;               // as the issuer's
    if constexpr (KIND == 1 && CG == 2) {
      // (all warps of the pair, whether their rows exist or not, go through the changes together: their arrivals are counted)
      bool go = true;
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int i = 0; i < HELD; ++i)
#pragma unroll
          for (int j = 0; j < COLS; ++j) held[m][i][j] = 0.f;
      auto take = [&](uint32_t& at, float (&sum)[HELD][COLS], int t) {
        if (go) go = __all_sync(0xffffffffu, wait(turn_full, (uint32_t)t & 1u, 245));
        if (go && live) {
          tc_fence_after();
          float v[HELD][COLS];
#pragma unroll
          for (int i = 0; i < HELD; ++i) tmem_ld16_nowait(at + (uint32_t)((part + i * kParts) * COLS), reinterpret_cast<uint32_t*>(v[i]));
          tmem_ld_wait();
          tc_fence_before();
#pragma unroll
          for (int i = 0; i < HELD; ++i)
#pragma unroll
            for (int j = 0; j < COLS; ++j) sum[i][j] += v[i][j];
        }
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(mapa_u32(smem_u32(&turn_done), 0));
        const uint32_t done = at;
        at = spare;
        spare = done;
      };
      for (int t = 0; t < p.turns; t += 2) {
        take(at0, held[0], t);
        if (t + 1 < p.turns) take(at1, held[1], t + 1);
      }
      live = live && go;
    }
    if (live && __all_sync(0xffffffffu, wait(acc_full, 0, 243))) {
      tc_fence_after();
      // two blocks of eight columns of all chains
      auto load = [&](uint32_t c0, uint32_t c1, float* v) {
        auto fetch = [&](int chain, float* t) {
          const uint32_t at = lanes + (uint32_t)chain * p.acc_cols;
          if constexpr (KIND == 2 && CG == 2) {
            tmem_ld8_nowait(at + c0, reinterpret_cast<uint32_t*>(t));
            tmem_ld8_nowait(at + c1, reinterpret_cast<uint32_t*>(t + 8));
          } else {
            tmem_ld16_nowait(at + c0, reinterpret_cast<uint32_t*>(t));              // (c1 is c0 + 8)
          }
        };
        float t[COLS], u[COLS];
        fetch(0, v);
        if (p.chains > 1) fetch(1, t);
        if (p.chains > 2) fetch(2, u);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < COLS; ++j) v[j] += (p.chains > 1 ? t[j] : 0.f) + (p.chains > 2 ? u[j] : 0.f);
        if (p.chains > 3) {
          fetch(3, t);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < COLS; ++j) v[j] += t[j];
        }
        if constexpr (MANY) {
#pragma unroll 1
          for (int chain = 4; chain < p.chains; chain += 2) {
            fetch(chain, t);
            if (chain + 1 < p.chains) fetch(chain + 1, u);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < COLS; ++j) v[j] += t[j] + (chain + 1 < p.chains ? u[j] : 0.f);
          }
        }
      };
      if constexpr (KIND == 1) {
        auto finish = [&](int c, float* v) {
          int g[2];
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            int lg = 2 * c + half, r = 0;                    // the column group's place among its CTA's, and which CTA that is
            if constexpr (CG == 2) {
              const int base = !turning || c < kTurnGroups ? 0 : c < 2 * kTurnGroups ? kTurnGroups : 2 * kTurnGroups;
              const int here = turning && c < 2 * kTurnGroups ? kTurnGroups : p.groups - base;
              lg -= 2 * base;
              r = lg >= here ? 1 : 0;
              lg += base - r * here;
            }
            g[half] = 2 * c + half < CG * p.groups ? group0 + lg + (r - rank) * p.groups : p.F;
          }
          uint2 o[2];
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            float* a = v + 8 * half;
            float x[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) x[j] = a[j] / (1.0f + expf(-a[j])) * a[4 + j];
            o[half] = make_uint2(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]));
          }
          if (!ok) return;
          bf16* at = p.act + (size_t)row * p.F;
          // (a store instruction costs the lines it touches, and every lane has a row of its own: the fewer the better)
          if (g[1] == g[0] + 1 && !(g[0] & 1) && 4 * g[1] < p.F) {
            *reinterpret_cast<uint4*>(at + 4 * g[0]) = make_uint4(o[0].x, o[0].y, o[1].x, o[1].y);
          } else {
            if (4 * g[0] < p.F) *reinterpret_cast<uint2*>(at + 4 * g[0]) = o[0];
            if (4 * g[1] < p.F) *reinterpret_cast<uint2*>(at + 4 * g[1]) = o[1];
          }
        };
        if (CG == 2 && turning) {
#pragma unroll
          for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int i = 0; i < (CG == 2 ? HELD : 1); ++i) {
              const int c = part + i * kParts;
              float v[COLS];
              tmem_ld16_nowait((m ? at1 : at0) + (uint32_t)(c * COLS), reinterpret_cast<uint32_t*>(v));
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < COLS; ++j) v[j] += held[m][i][j];
              finish(c + m * kTurnGroups, v);
            }
          const int rest = p.groups - 2 * kTurnGroups;
          for (int c = part; c < rest; c += kParts) {
            float v[COLS], t[COLS];
            const uint32_t from = lanes + (uint32_t)(3 * kTurnCols + c * COLS);
            tmem_ld16_nowait(from, reinterpret_cast<uint32_t*>(v));
            tmem_ld16_nowait(from + (uint32_t)(rest * COLS), reinterpret_cast<uint32_t*>(t));
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < COLS; ++j) v[j] += t[j];
            finish(c + 2 * kTurnGroups, v);
          }
        } else {
          for (int c = part; 2 * c < CG * p.groups; c += kParts) {
            float v[COLS];
            load((uint32_t)(c * COLS), (uint32_t)(c * COLS + 8), v);
            finish(c, v);
          }
        }
      } else if constexpr (KIND == 0) {
        for (int c = part; 2 * c < CG * p.groups; c += kParts) {
          float v[COLS];
          load((uint32_t)(c * COLS), (uint32_t)(c * COLS + 8), v);
          const int n = (tile * CG * p.groups + 2 * c) * 8, cols = min(2 * c + 2 <= CG * p.groups ? 16 : 8, p.N - n);
          float* o = p.out + ((size_t)slot * p.M + row) * p.N + n;
          if (!ok) continue;
          if (!(p.N & 3)) {
#pragma unroll
            for (int j = 0; j < COLS; j += 4)
              if (j < cols) *reinterpret_cast<float4*>(o + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
          } else {
#pragma unroll
            for (int j = 0; j < COLS; ++j)
              if (j < cols) o[j] = v[j];
          }
        }
      } else {
        // a step: two heads of this CTA, or a head's rotations of both CTAs (next to each other)
        const RopeEpilogue& e = p.re;
        for (int c = part; CG == 2 ? c < p.groups : 2 * c < p.groups; c += kParts) {
          float v[COLS];
          if constexpr (CG == 2) load((uint32_t)(c * 8), (uint32_t)((p.groups + c) * 8), v);
          else load((uint32_t)(c * COLS), (uint32_t)(c * COLS + 8), v);
          uint2 lo[2], hi[2];
          bf16* o[2];
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            const int lg = CG == 2 ? c : 2 * c + half, r = CG == 2 ? half : 0, g = group0 + lg;
            const int which = g / e.H, h = g - which * e.H;
            float* a = v + 8 * half;
            float* b = a + 4;
            if (which < 2)
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const float o1 = a[j] * cs[r][j] - b[j] * sn[r][j];
                b[j] = b[j] * cs[r][j] + a[j] * sn[r][j];
                a[j] = o1;
              }
            lo[half] = make_uint2(pack_bf16(a[0], a[1]), pack_bf16(a[2], a[3]));
            hi[half] = make_uint2(pack_bf16(b[0], b[1]), pack_bf16(b[2], b[3]));
            o[half] = !ok || lg >= p.groups || which > 2 ? nullptr
                      : which == 0 ? reinterpret_cast<bf16*>(e.q) + ((size_t)row * e.H + h) * 128
                                   : reinterpret_cast<bf16*>(which == 1 ? e.kpool : e.vpool) + (kv + (size_t)h * CERB_PAGE) * 128;
          }
          if constexpr (CG == 2) {
            if (o[0]) {
              bf16* at = o[0] + (row0 & ~7);
              *reinterpret_cast<uint4*>(at) = make_uint4(lo[0].x, lo[0].y, lo[1].x, lo[1].y);
              *reinterpret_cast<uint4*>(at + 64) = make_uint4(hi[0].x, hi[0].y, hi[1].x, hi[1].y);
            }
          } else {
#pragma unroll
            for (int half = 0; half < 2; ++half)
              if (o[half]) {
                *reinterpret_cast<uint2*>(o[half] + row0) = lo[half];
                *reinterpret_cast<uint2*>(o[half] + row0 + 64) = hi[half];
              }
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (p.clk && threadIdx.x == 0) atomicMax(p.clk + kGemmClockSlots, globaltimer_ns());
  if constexpr (CG == 2) {
    // Neither CTA leaves (nor frees its tensor memory) before the other is done: copies, commits and arrivals cross between them until then.
    if (warp == 2) cluster_meet_before_exit(&meet_bar, 2, lane, wc, &meet_flag_s, 246);
    __syncthreads();
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
  } else {
    if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(p.tmem_cols) : "memory");
  }
}

template <int KIND, int CG, bool MANY>
int launch_kind(const CUtensorMap& tmW, const CUtensorMap& tmX, const RowsParams& p, int tiles, cudaStream_t st) {
  auto kern = gemm_rows_kernel<KIND, CG, MANY>;
  static std::atomic<bool> configured{false};
  if (!configured) {
    CERB_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRing));
    configured = true;
  }
  // (always the same request, more than half of an SM: one CTA there, which may own all of its tensor memory)
  const cudaError_t e = CG == 2 ? launch_pdl_cluster(kern, dim3((tiles + 1) / 2 * 2), dim3(kThreads), kRing, st, 2u, tmW, tmX, p)
                                : launch_pdl(kern, dim3(tiles), dim3(kThreads), kRing, st, tmW, tmX, p);
  return e == cudaSuccess ? CERB_OK : CERB_E_CUDA;
}

// (activation tiles of 16 or 48 rows: forwards 2 % slower than with 32 and 64)
size_t rows_fetched(int M) { return ((M > ROWS ? (M + 1) / 2 : M) + 31) / 32 * 32; }
// Up to 64 rows: MMAs of 64 rows.  A stream of weights at the HBM rate and half-empty MMAs run into the power limit together: 64-node forwards of the 7B
// shape, one after the other, 3511 us with MMAs of 128 rows and 3358 with 64; the first ones on an idle GPU take 3280 either way.
int mma_rows(int M) { return M <= 64 ? 64 : ROWS; }
int acc_columns(const RowsPlan& g, int M) {
  const int step = mma_rows(M) == 64 ? 8 : 16;
  return (g.groups * 8 * (M > ROWS ? 2 : 1) + step - 1) / step * step;
}
int ring_stages(const RowsPlan& g, int M) {
  const size_t stage = (size_t)g.groups * 1024 + rows_fetched(M) * 128;
  // (the MMAs read all rows of the last stage, too; 1 KB for the alignment of the ring)
  const int stages = (int)((kRing - 1024 - (mma_rows(M) - rows_fetched(M)) * 128) / stage);
  return stages < MAX_STAGES ? stages : MAX_STAGES;
}
Chains ring_chains(const RowsPlan& g, const RowsRing& r, int num_kb) {
  Chains c;
  const int parts = g.parts ? g.parts : 1;
  for (int s = 0; s < parts; ++s) {
    const int n = (s + 1) * num_kb / parts - s * num_kb / parts;
    for (int i = 0; i < r.issuers; ++i) c.add((n - i + r.issuers - 1) / r.issuers, (r.chains - i + r.issuers - 1) / r.issuers);
  }
  return c;
}
// What runs a plan's product of up to `limit` rows: the ring, the issuers, and as many accumulators as its chains need to be no longer than `other`.
// A stage belongs to one issuer, which waits for its phases in turn.  (Issuers that took turns at a stage could be a round apart when copies
// land out of order, and a parity tells neighbouring phases apart only.)  Three issuers or two where the ring loses no stage by it; one
// where it would and the weights of a stage take as long to come as one issuer needs.
RowsRing plan_ring(const RowsPlan& g, int limit, int K, const Chains& other) {
  const int num_kb = (K + BK - 1) / BK, least_kb = g.parts ? num_kb / g.parts : num_kb, cols = acc_columns(g, limit);
  RowsRing r;
  r.stages = ring_stages(g, limit);
  r.issuers = r.stages % 3 == 0 && 3 * cols <= 512 ? 3 : r.stages % 2 == 0 ? 2 : g.groups >= 16 ? 1 : 2;
  r.stages -= r.stages % r.issuers;
  if (r.issuers > least_kb) r.issuers = least_kb;
  const int most = 512 / cols < least_kb ? 512 / cols : least_kb;
  r.chains = r.issuers < 3 && 2 * r.issuers <= most ? 2 * r.issuers : r.issuers;
  while (r.chains <= most && !ring_chains(g, r, num_kb).no_longer_than(other)) ++r.chains;
  if (r.chains > most) r.chains = 0;
  return r;
}

}  // namespace

Chains gemm_rows_other_chains(int limit, int N, int K) {
  if (limit <= ROWS) return gemm_bf16_chains(N, K);
  const Chains a = gemm_tile_chains(limit - 32, N, K), b = gemm_tile_chains(limit, N, K);
  return a.no_longer_than(b) ? a : b;
}

namespace {

// Three MMAs per 16 k: a change of accumulators every eighth of k
int turn_blocks(int num_kb) { return num_kb / 8; }
int turn_count(int num_kb) { return (num_kb - 1) / turn_blocks(num_kb); }
bool turns_fit(const RowsPlan& g, int K) {
  return 3 * kTurnCols + 2 * (16 * g.groups - 2 * kTurnCols) <= 512 && (K + BK - 1) / BK >= 16;
}
Chains turn_chains(const RowsPlan& g, int num_kb) {
  Chains c;
  for (int column = 0; column < g.groups; ++column)                // (16 columns at a time)
    if (column < 2 * kTurnGroups) {
      int since = 0;
      for (int t = column / kTurnGroups; t < turn_count(num_kb); t += 2) {
        c.chain((t + 1) * turn_blocks(num_kb) - since);
        since = (t + 1) * turn_blocks(num_kb);
      }
      c.chain(num_kb - since);
    } else {
      c.add(num_kb, 2);
    }
  return c;
}
void plan_rings(RowsPlan& g, int N, int K) {
  for (int i = 0; i < kRowsClasses; ++i) {
    const int limit = rows_class_limit(i);
    if (g.heads && limit > ROWS && limit <= 192) continue;
    if (limit > ROWS && g.groups > 16) {
      if (g.heads || !turns_fit(g, K) || !turn_chains(g, (K + BK - 1) / BK).no_longer_than(gemm_rows_other_chains(limit, N, K))) continue;
      g.ring[i] = RowsRing{ring_stages(g, limit), 2, 5};
    } else {
      g.ring[i] = plan_ring(g, limit, K, gemm_rows_other_chains(limit, N, K));
    }
  }
}

}  // namespace

RowsPlan plan_rows_swiglu(int F, int K) {
  RowsPlan g{};
  const int groups = F / 4, per = (groups + kSms - 1) / kSms;
  if (F % 4 || per < 2 || per > 32) return g;
  g.groups = per;
  g.tiles = (groups + per - 1) / per;
  plan_rings(g, 2 * F, K);
  return g;
}

RowsPlan plan_rows_rope(int n_heads, int head_dim, int K) {
  RowsPlan g{};
  g.heads = true;
  const int heads = 3 * n_heads, per = (heads + kSms / 16 - 1) / (kSms / 16);
  if (head_dim != 128 || per < 2 || per > 32) return g;
  g.groups = per;
  g.tiles = 16 * ((heads + per - 1) / per);
  plan_rings(g, heads * 128, K);
  return g;
}

// Which products come here, from 9 rows on.
//   Up to 128 rows, against partial sums and kernels behind them: matrices of at least 16 rows per SM (an MMA's N is no less) and at most 256.
//   Forwards, plain sums (below) included: 7B width 9 / 64 / 128 rows 1.06 / 1.06 / 1.12 x, 13B 1.02 / 1.09 / 1.13 x, 1024 to 3200 columns 1.04 to 1.25 x.
//   129 to 256 rows, in pairs, against output tiles of 256 weight rows (gemm_tile.cu): a pair's tile has to fit one MMA, or (SwiGLU, 16 k
//   blocks and more, up to 304 columns) three as above.  Tiles of 256 rows leave SMs idle or have to be cut along k: 7B width, gate-up of 129 / 256 rows 46 / 53 -> 41 /
//   43 us with two MMAs a tile, and 1 us more with three (as above).  RoPE from 193 rows on: below, the output tiles are cut and sum shorter chains than those that fit here (keys of 130 to 180 rows against float64
//   1.10e-4 to 1.32e-4 there, 1.32e-4 to 1.52e-4 here).  From 193 rows on they are as long at 4096 columns and more (QKV of 256 rows 32.5 -> 27 us) and fit at 1024
//   and 1536; from 2048 to 3584 they do not (2048 columns, 2 x 128 rows, 8 layers: 580 us here, 645 with output tiles; V 0.44 against 0.24e-6 from float64).
bool gemm_rows_takes(const RowsPlan& g, int M) {
  const int i = rows_class(M);
  return i >= 0 && g.tiles > 0 && g.ring[i].chains > 0;
}

Chains gemm_rows_chains(const RowsPlan& g, int M, int K) {
  const RowsRing& r = g.ring[rows_class(M)];
  const int num_kb = (K + BK - 1) / BK;
  return M > ROWS && g.groups > 16 ? turn_chains(g, num_kb) : ring_chains(g, r, num_kb);
}

// Plain sums of up to 128 rows (O, down, LM head): k is cut into parts, each a sum of its own (a slot) for the kernel behind to add, so that tiles are wide
// enough.  A CTA takes in its weights (8 x groups rows) at 44 bytes a ns, its share of the HBM rate, and everything, activations included, at
// 85; a k block takes 0.34 us, however narrow the tile.  7B width, 64 rows, 8 layers: down in 2 / 4 / 5 / 8 parts 872 / 847 / 845 / 859 us, O in 4 / 5 / 8
// 847 / 845 / 856.  (Units of 256 weight rows left ten slots after both, 10 MB that the norm read back; slots of the same plan, 64 rows: norm 4.65 ->
// 4.0 us, O 9.8 -> 8.8, down 17.6 -> 16.5.)
// 129 to 256 rows, in pairs: the same, a part costing more (4 MB to write and to read back at 256 rows and 4096 columns).
RowsPlan plan_rows_sums(int M, int N, int K, int max_parts) {
  RowsPlan best{};
  double best_t = 0;
  const int pair = M > ROWS ? 2 : 1, groups = (N + 7) / 8, num_kb = (K + BK - 1) / BK, x = ((M + pair - 1) / pair + 31) / 32 * 32 / 8;
  if (M <= kFewRows || M > 2 * ROWS) return best;
  for (int parts = 1; parts <= max_parts && parts <= 8 && parts * 4 <= num_kb; ++parts) {
    const int tiles = kSms / pair / parts, per = (groups + pair * tiles - 1) / (pair * tiles);
    if (per > 32 / pair || per < 2) continue;
    const double kb = (num_kb + parts - 1) / parts;
    const double hbm = kb * per / 44.0, sm = kb * (per + x) / 85.0;
    const double least = kb * 0.34;                      // a stage's copies, waits and MMAs
    const double in = hbm > sm ? hbm : sm, t = (in > least ? in : least) + parts * (pair == 2 ? 0.004 * M : 0.05 + 0.001 * M);
    if (!best_t || t < best_t) {
      best_t = t;
      best = RowsPlan{per, (groups + pair * per - 1) / (pair * per) * parts * pair, false, parts, {}};
    }
  }
  if (!best.tiles) return best;
  RowsRing& r = best.ring[rows_class(M)];
  r = plan_ring(best, M, K, gemm_rows_other_chains(M, N, K));
  return r.chains ? best : RowsPlan{};
}

int launch_gemm_rows(cerb_ctx* c, const CUtensorMap* tmW, const ActMaps* tmX, const RowsPlan& g, int M, int N, int K, int32_t* status, cudaStream_t st,
                     const GemmEpilogue* epi, float* out, unsigned long long* clock_slot) {
  const int i = rows_class(M);
  if (i < 0 || !g.ring[i].chains || (!epi && g.parts < 1)) return CERB_E_SHAPE;
  const bool pairs = M > ROWS;            // (7B width, 96 and 128 rows: 1062 and 1082 us in pairs, 926 and 974 in single CTAs)
  RowsParams p;
  memset(&p, 0, sizeof(p));
  p.status = status;
  p.M = M;
  p.F = N / 2;
  p.num_kb = (K + BK - 1) / BK;
  p.out = out;
  p.N = N;
  p.parts = g.parts;
  p.groups = g.groups;
  p.x_rows = (int)rows_fetched(M);
  p.m_rows = mma_rows(M);
  p.stages = g.ring[i].stages;
  p.issuers = g.ring[i].issuers;
  p.chains = g.ring[i].chains;
  if (pairs && g.groups > 16) {
    p.turn = turn_blocks(p.num_kb);
    p.turns = turn_count(p.num_kb);
    p.tmem_cols = 512;
  } else {
    p.acc_cols = (uint32_t)acc_columns(g, M);
    for (p.tmem_cols = 32; p.tmem_cols < p.chains * p.acc_cols; p.tmem_cols *= 2) {}
  }
  p.wait_cycles = wait_cycles();
  p.clk = clock_slot;
  auto run = [&](auto kind, const CUtensorMap& x) {
    constexpr int KIND = decltype(kind)::value;
    if (p.chains > 4 && !p.turns) return pairs ? launch_kind<KIND, 2, true>(*tmW, x, p, g.tiles, st) : launch_kind<KIND, 1, true>(*tmW, x, p, g.tiles, st);
    return pairs ? launch_kind<KIND, 2, false>(*tmW, x, p, g.tiles, st) : launch_kind<KIND, 1, false>(*tmW, x, p, g.tiles, st);
  };
  int rc;
  if (!epi) {
    rc = run(std::integral_constant<int, 0>(), tmX->box(p.x_rows));
  } else if (epi->kind == 1) {
    p.act = (bf16*)epi->act;
    rc = run(std::integral_constant<int, 1>(), tmX->box(p.x_rows));
  } else {
    p.re = *epi->rope;
    rc = run(std::integral_constant<int, 2>(), tmX->box(p.x_rows));
  }
  if (rc != CERB_OK) return rc;
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

}  // namespace cerb
