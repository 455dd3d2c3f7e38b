// Tree-verification attention (Sections 1 and 3.1: all candidates are verified in one pass with
// tree attention).  Query i of a sequence sees every committed prefix key and those tree keys j
// that are its ancestors (bit j of anc[i]), nothing else.
//
// bf16 path: one CTA per (split, head, sequence).  A producer warp streams 64-key tiles (four
// 16-token pages of one head, K and V) into shared memory with TMA, 128-byte swizzled, through an
// mbarrier ring; compute warps run QK^T and PV on tensor cores (warp-level MMA, fp32 accumulate)
// with an online softmax in registers.  Warps are arranged WQ x WK: WQ blocks of 16 query rows,
// WK slices of each key tile, so small trees still use every warp.  Long contexts are split along
// the keys; each split writes an unnormalised partial (m, l, O) and the last CTA to finish for a
// (sequence, head) merges the partials in split order, so the result does not depend on timing.
//
// fp32 path (CERB_F32 models): plain FMA arithmetic, one CTA per (node, head, sequence).
#include <stdlib.h>

#include <atomic>

#include "tc_common.cuh"

namespace cerb {

namespace {

constexpr int TILE = 64;                  // keys per pipeline stage = 4 pages
constexpr int PAGES_PER_TILE = TILE / CERB_PAGE;
constexpr int kTargetCtas = 296;          // two CTAs per SM on a 148-SM part
constexpr int kMaxSplit = 32;
constexpr int kMaxPagesPerCta = 1024;
constexpr size_t kCounterBytes = 4096;    // one ticket counter per (sequence, head)
constexpr int kAttnRowsPerLaunch = 128;   // query rows a CTA holds at most

// K/V tiles are read once per step (the next layer's tiles, and 13 GB of weights, come before they are needed
// again): they enter L2 with evict-first priority so that they do not push out activations and partial sums.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  tma_load_2d_hint(dst, map, x, y, bar, l2_policy(true));
}
__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t& r0, uint32_t& r1, uint32_t& r2, uint32_t& r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(addr));
}
__device__ __forceinline__ void mma_bf16(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void compute_bar(int nthreads) { asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory"); }

// Which of the 64 keys key0 .. key0 + 63 one query row may see, as a bit mask (bit j <-> key key0 + j): prefix keys
// (position < L) always, tree keys by the row's ancestor words a0, a1, a2 (tree index = position - L).  Ancestor
// words have no bits at or above the live node count, so keys past the last live tree key come out invisible.
// Called only for tiles that reach past the prefix (key0 + 64 > L).
__device__ __forceinline__ uint64_t tile_visibility(int key0, int L, uint64_t a0, uint64_t a1, uint64_t a2) {
  const int base = key0 - L;                       // tree index of the tile's first key; negative: the tile starts in the prefix
  if (base < 0) {
    const int s = -base;                           // 1 .. 63 prefix keys, then tree keys 0 .. 63 - s
    return (a0 << s) | ((1ull << s) - 1ull);
  }
  const int w = base >> 6, sh = base & 63;
  const uint64_t lo = w == 0 ? a0 : w == 1 ? a1 : w == 2 ? a2 : 0ull;
  const uint64_t hi = w == 0 ? a1 : w == 1 ? a2 : 0ull;
  return sh ? (lo >> sh) | (hi << (64 - sh)) : lo;
}

struct AttnParams {
  const bf16* q;
  const int32_t* page_table;
  const int32_t* len;
  const int32_t* n_active;
  const uint64_t* anc;
  const int32_t* row_off;   // first row of every sequence in q / out, or null: sequence b starts at row b * n
  bf16* out;
  float* lse;
  float* partial;           // [B*H][nsplit][NQ][DH+4]
  unsigned int* counters;   // [B*H]
  int32_t* status;
  int n, H, max_pages, nsplit, oob_row;
  int B, Bw;                // sequences; (sequence, window) pairs
  int win, win0;            // a prefill chunk of consecutive tokens per sequence: its windows of 128 query rows win0 .. win0 + win - 1, one
                            // per blockIdx.z (locate_window); 1 and 0 otherwise
  int row0, rows;           // query rows row0 .. row0 + rows - 1 of the tree are this launch's (q, out, lse and anc already point
                            // at row0); a tree of more than 128 nodes takes two launches.  n stays the tree's node count
                            // (the row stride between sequences); only keys below row0 + rows can be ancestors of these rows.
  int rows_pad;             // rows per split in `partial` (16, 32, 64 or 128)
  uint32_t v_lbo, v_sbo;    // byte offsets of the V operand's descriptor (tensor-core path)
  long long wait_cycles;    // budget of every bounded wait, SM clock cycles
  int cluster;              // tensor-core path: the splits of a (sequence, head) form one cluster and merge through shared memory
  float scale_log2;
  int items, item0;         // tensor-core kernels, PART: the launch's (sequence or window, head) items, and the first of them
  int follows;              // ... the launch in front is of the same call: it writes nothing that this one reads and reads nothing that this one
                            // writes.  What that one waited for is complete, so this one waits (and lets its own dependents go) only at its end.
};

// Which sequence, and which window of 128 query rows of it, z (blockIdx.z in most kernels) stands for.  A prefill chunk is one long
// chain: window w is a chain of 128 nodes behind `shift` = 128 w more prefix keys, all of them in the cache before this
// launch.  The last windows see the most keys and come first, so that the short ones fill the launch's tail.
__device__ __forceinline__ void locate_window(const AttnParams& p, int z, int& b, int& shift) {
  b = p.win > 1 ? z % p.B : z;
  shift = (p.win0 + (p.win > 1 ? p.win - 1 - z / p.B : 0)) * kAttnRowsPerLaunch;
}

template <int DH, int WQ, int WK, int STAGES>
__global__ void __launch_bounds__((WQ * WK + 1) * 32) tree_attn_bf16_kernel(const __grid_constant__ CUtensorMap tmK,
                                                                          const __grid_constant__ CUtensorMap tmV,
                                                                          const AttnParams p) {
  constexpr int NW = WQ * WK;               // compute warps
  constexpr int NQ = WQ * 16;               // query rows of this CTA
  constexpr int KW = TILE / WK;             // keys per warp per tile
  constexpr int NT = KW / 8;                // 8-key score tiles per warp
  constexpr int HALVES = DH / 64;
  constexpr uint32_t HALF_BYTES = TILE * 128;
  constexpr uint32_t KV_BYTES = HALVES * HALF_BYTES;      // one of K or V for a stage
  constexpr uint32_t STAGE_BYTES = 2 * KV_BYTES;
  constexpr int ROWF = DH + 4;                            // merge row: O[DH], m, l, pad (16-byte rows)
  static_assert(NQ * ROWF * 4 <= STAGES * STAGE_BYTES, "merge buffer must fit in the stage ring");

  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[STAGES];
  __shared__ __align__(8) uint64_t empty_bar[STAGES];
  __shared__ int page_list[kMaxPagesPerCta];
  __shared__ int aborted_s, exit_flag_s;
  __shared__ unsigned int ticket_s;
  __shared__ __align__(8) uint64_t cl_bar[2];
  volatile int* aborted = &aborted_s;
  const WaitCtx wc{p.wait_cycles, aborted, p.status};

  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  // Lengths, live node counts, the page table and the prefix keys were written at least two kernels ago:
  // set-up, the page list and the first prefix tiles run before griddep_wait() and overlap the previous
  // kernel's tail; Q and this step's tree keys are only touched after it.
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int split = blockIdx.x, h = blockIdx.y;
  int b, shift;
  locate_window(p, (int)blockIdx.z, b, shift);
  const int L_old = p.len[b], L = L_old + shift;                      // keys written by earlier launches; keys every row sees
  const int nq_all = (p.n_active ? min(p.n_active[b], p.n) : p.n) - shift;   // live nodes of this sequence (from the window on)
  const size_t qrow = (p.row_off ? (size_t)p.row_off[b] : (size_t)b * p.n) + shift;   // its first row of q and out
  const int nq = min(nq_all - p.row0, p.rows);                        // live query rows of this launch
  if (nq <= 0) {
    griddep_wait();      // (no CTA leaves ahead of the kernel in front: this launch would count as complete while that one runs)
    return;
  }
  const int kv_total = L + min(nq_all, p.row0 + p.rows);
  const int tiles = (kv_total + TILE - 1) / TILE;
  const int per = (tiles + p.nsplit - 1) / p.nsplit;
  const int t0 = min(tiles, split * per), t1 = min(tiles, t0 + per);
  const bool too_long = per * PAGES_PER_TILE > kMaxPagesPerCta;

  if (threadIdx.x == 0) {
    aborted_s = (*p.status != 0);
    exit_flag_s = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), NW);
    }
    mbar_init(smem_u32(&cl_bar[0]), (uint32_t)p.nsplit);
    mbar_init(smem_u32(&cl_bar[1]), (uint32_t)p.nsplit);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (too_long) atomicExch(p.status, CERB_E_SHAPE);
  }
  __syncthreads();
  if (p.cluster) cluster_start_arrive();
  const int t_end = too_long ? t0 : t1;

  float* mrg = reinterpret_cast<float*>(smem_gen);   // [NQ][ROWF], used after the key loop

  if (warp == NW) {
    // ---------------- producer warp ----------------
    const int32_t* pt = p.page_table + (size_t)b * p.max_pages;
    const int n_pages = (t_end - t0) * PAGES_PER_TILE;
    for (int i = lane; i < n_pages; i += 32) {
      int lp = t0 * PAGES_PER_TILE + i;
      page_list[i] = (lp * CERB_PAGE < kv_total && lp < p.max_pages) ? (pt[lp] * p.H + h) * CERB_PAGE : p.oob_row;
    }
    __syncwarp();
    if (lane == 0) {
      int early = 0;
      while (t0 + early < t_end && early < STAGES && (t0 + early + 1) * TILE <= L_old) ++early;
      // (the abort flag itself is looked at once, for a launch that starts after a time-out: nothing is issued then;
      // later a wait that gives up says so in its return value, which costs the loop nothing)
      const int t_stop = *aborted ? t0 : t_end;
      int i = 0;
      for (int t = t0; t < t_stop; ++t, ++i) {
        if (i == early) { griddep_wait(); griddep_launch(); }
        int s = i % STAGES;
        uint32_t ph = (uint32_t)(i / STAGES) & 1u;
        if (!mbar_wait(smem_u32(&empty_bar[s]), ph ^ 1u, wc, 301)) break;      // the consumers have stopped: issue nothing more
        uint32_t fb = smem_u32(&full_bar[s]);
        mbar_expect_tx(fb, STAGE_BYTES);
        uint32_t kdst = smem_base + (uint32_t)s * STAGE_BYTES, vdst = kdst + KV_BYTES;
#pragma unroll
        for (int pg = 0; pg < PAGES_PER_TILE; ++pg) {
          int row = page_list[i * PAGES_PER_TILE + pg];      // out-of-range rows are zero-filled by TMA
#pragma unroll
          for (int hf = 0; hf < HALVES; ++hf) {
            uint32_t off = (uint32_t)hf * HALF_BYTES + (uint32_t)pg * (CERB_PAGE * 128);
            tma_load_2d(kdst + off, &tmK, hf * 64, row, fb);
            tma_load_2d(vdst + off, &tmV, hf * 64, row, fb);
          }
        }
      }
      if (*aborted) {
        // give-up path: the copies already issued (units 0 .. i-1) still land in this CTA's shared memory; see each of them in
        for (int j = i > STAGES ? i - STAGES : 0; j < i; ++j)
          mbar_wait_drain(smem_u32(&full_bar[j % STAGES]), (uint32_t)(j / STAGES) & 1u, 20000000ll);
      }
    }
    griddep_wait();      // (a lane that has waited already returns at once)
    griddep_launch();
  } else {
    // ---------------- compute warps ----------------
    griddep_wait();
    griddep_launch();
    const int qi = warp % WQ, ki = warp / WQ;
    const int g = lane >> 2, tq = lane & 3;
    const int r0 = qi * 16 + g, r1 = r0 + 8;                // this thread's two query rows
    // Q fragments straight from global memory (A operand of m16n8k16, one per 16 head-dim elements)
    uint32_t qa[DH / 16][4];
    {
      const bf16* q0 = p.q + ((qrow + r0) * p.H + h) * DH;
      const bf16* q1 = p.q + ((qrow + r1) * p.H + h) * DH;
#pragma unroll
      for (int kk = 0; kk < DH / 16; ++kk) {
        int c = kk * 16 + tq * 2;
        qa[kk][0] = r0 < nq ? *reinterpret_cast<const uint32_t*>(q0 + c) : 0u;
        qa[kk][1] = r1 < nq ? *reinterpret_cast<const uint32_t*>(q1 + c) : 0u;
        qa[kk][2] = r0 < nq ? *reinterpret_cast<const uint32_t*>(q0 + c + 8) : 0u;
        qa[kk][3] = r1 < nq ? *reinterpret_cast<const uint32_t*>(q1 + c + 8) : 0u;
      }
    }
    uint64_t anc0[CERB_ANC_WORDS], anc1[CERB_ANC_WORDS];
#pragma unroll
    for (int w = 0; w < CERB_ANC_WORDS; ++w) {
      anc0[w] = r0 < nq ? p.anc[r0 * CERB_ANC_WORDS + w] : 0ull;
      anc1[w] = r1 < nq ? p.anc[r1 * CERB_ANC_WORDS + w] : 0ull;
    }

    float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
    float o[DH / 8][4];
#pragma unroll
    for (int i = 0; i < DH / 8; ++i) { o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f; }

    for (int t = t0, it = 0; t < t_end; ++t, ++it) {
      const int s = it % STAGES;
      const uint32_t ph = (uint32_t)(it / STAGES) & 1u;
      mbar_wait(smem_u32(&full_bar[s]), ph, wc, 302);
      const uint32_t kbase = smem_base + (uint32_t)s * STAGE_BYTES, vbase = kbase + KV_BYTES;
      const int key_tile0 = t * TILE;
      if (key_tile0 + TILE > kv_total) {
        // last, partial tile: rows past the end may hold anything (stale pool memory); zero V there so
        // that a zero probability times a non-finite value cannot poison the sum.
        const int first_bad = kv_total - key_tile0;
        uint8_t* vgen = smem_gen + (size_t)s * STAGE_BYTES + KV_BYTES;
        for (int idx = warp * 32 + lane; idx < (TILE - first_bad) * HALVES * 8; idx += NW * 32) {
          int row = first_bad + idx / (HALVES * 8), rem = idx % (HALVES * 8);
          *reinterpret_cast<uint4*>(vgen + (size_t)(rem / 8) * HALF_BYTES + row * 128 + (rem % 8) * 16) = make_uint4(0, 0, 0, 0);
        }
        compute_bar(NW * 32);
      }

      // ---- S = Q K^T for this warp's key slice ----
      float sc[NT][4];
#pragma unroll
      for (int i = 0; i < NT; ++i) { sc[i][0] = sc[i][1] = sc[i][2] = sc[i][3] = 0.f; }
      const int mat = lane >> 3, lr = lane & 7;
#pragma unroll
      for (int kk = 0; kk < DH / 16; ++kk) {
#pragma unroll
        for (int nt = 0; nt < NT; nt += 2) {
          int key = ki * KW + nt * 8 + (mat >> 1) * 8 + lr;
          int chunk = kk * 2 + (mat & 1);
          uint32_t addr = kbase + (uint32_t)(chunk >> 3) * HALF_BYTES + (uint32_t)key * 128 + (uint32_t)(((chunk & 7) ^ (key & 7)) << 4);
          uint32_t b0, b1, b2, b3;
          ldsm_x4(addr, b0, b1, b2, b3);
          mma_bf16(sc[nt], qa[kk][0], qa[kk][1], qa[kk][2], qa[kk][3], b0, b1);
          mma_bf16(sc[nt + 1], qa[kk][0], qa[kk][1], qa[kk][2], qa[kk][3], b2, b3);
        }
      }

      // ---- mask, online softmax ----
      const bool need_mask = key_tile0 + TILE > L;
      uint64_t vm0 = ~0ull, vm1 = ~0ull;             // visible keys of this tile for rows r0 and r1
      if (need_mask) {
        vm0 = tile_visibility(key_tile0, L, anc0[0], anc0[1], anc0[2]);
        vm1 = tile_visibility(key_tile0, L, anc1[0], anc1[1], anc1[2]);
      }
      float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float v = sc[nt][e] * p.scale_log2;
          if (need_mask) {
            const int j = ki * KW + nt * 8 + tq * 2 + (e & 1);          // key's index inside the tile
            if (!((((e < 2) ? vm0 : vm1) >> j) & 1ull)) v = -INFINITY;
          }
          sc[nt][e] = v;
          if (e < 2) mx0 = fmaxf(mx0, v); else mx1 = fmaxf(mx1, v);
        }
      }
      mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 1));
      mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, 2));
      mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 1));
      mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, 2));
      const float mn0 = fmaxf(m0, mx0), mn1 = fmaxf(m1, mx1);
      const float mu0 = mn0 == -INFINITY ? 0.f : mn0, mu1 = mn1 == -INFINITY ? 0.f : mn1;
      const float al0 = exp2f(m0 - mu0), al1 = exp2f(m1 - mu1);
      m0 = mn0; m1 = mn1;
      float rs0 = 0.f, rs1 = 0.f;
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        sc[nt][0] = exp2f(sc[nt][0] - mu0); sc[nt][1] = exp2f(sc[nt][1] - mu0);
        sc[nt][2] = exp2f(sc[nt][2] - mu1); sc[nt][3] = exp2f(sc[nt][3] - mu1);
        rs0 += sc[nt][0] + sc[nt][1];
        rs1 += sc[nt][2] + sc[nt][3];
      }
      l0 = l0 * al0 + rs0;
      l1 = l1 * al1 + rs1;
#pragma unroll
      for (int i = 0; i < DH / 8; ++i) { o[i][0] *= al0; o[i][1] *= al0; o[i][2] *= al1; o[i][3] *= al1; }

      // ---- O += P V ----
#pragma unroll
      // Probabilities enter the tensor core as two bf16 terms, p = p_hi + p_lo (about 16 significant
      // bits), so that the product is not limited by bf16's 8-bit significand: with near-uniform
      // attention over many keys a single bf16 term costs as much accuracy as all other roundings together.
      for (int j = 0; j < KW / 16; ++j) {
        uint32_t ah[4], al[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float p0 = sc[2 * j + (e >> 1)][(e & 1) * 2], p1 = sc[2 * j + (e >> 1)][(e & 1) * 2 + 1];
          __nv_bfloat162 hi = __floats2bfloat162_rn(p0, p1);
          float2 hf = __bfloat1622float2(hi);
          ah[e] = *reinterpret_cast<uint32_t*>(&hi);
          al[e] = pack_bf16(p0 - hf.x, p1 - hf.y);
        }
#pragma unroll
        for (int dn = 0; dn < DH / 8; dn += 2) {
          int key = ki * KW + j * 16 + (mat & 1) * 8 + lr;
          int chunk = dn + (mat >> 1);
          uint32_t addr = vbase + (uint32_t)(chunk >> 3) * HALF_BYTES + (uint32_t)key * 128 + (uint32_t)(((chunk & 7) ^ (key & 7)) << 4);
          uint32_t b0, b1, b2, b3;
          ldsm_x4_t(addr, b0, b1, b2, b3);
          mma_bf16(o[dn], ah[0], ah[1], ah[2], ah[3], b0, b1);
          mma_bf16(o[dn + 1], ah[0], ah[1], ah[2], ah[3], b2, b3);
          mma_bf16(o[dn], al[0], al[1], al[2], al[3], b0, b1);
          mma_bf16(o[dn + 1], al[0], al[1], al[2], al[3], b2, b3);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&empty_bar[s]));
    }

    // ---- combine the WK key slices of each query block, through shared memory ----
    l0 += __shfl_xor_sync(0xffffffffu, l0, 1); l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
    l1 += __shfl_xor_sync(0xffffffffu, l1, 1); l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
    compute_bar(NW * 32);                       // every warp is done with the stage ring
    for (int kslice = 0; kslice < WK; ++kslice) {
      if (ki == kslice) {
        float* row0 = mrg + (size_t)r0 * ROWF;
        float* row1 = mrg + (size_t)r1 * ROWF;
        if (kslice == 0) {
#pragma unroll
          for (int i = 0; i < DH / 8; ++i) {
            int c = i * 8 + tq * 2;
            row0[c] = o[i][0]; row0[c + 1] = o[i][1]; row1[c] = o[i][2]; row1[c + 1] = o[i][3];
          }
          if (tq == 0) { row0[DH] = m0; row0[DH + 1] = l0; row1[DH] = m1; row1[DH + 1] = l1; }
        } else {
          float pm0 = row0[DH], pl0 = row0[DH + 1], pm1 = row1[DH], pl1 = row1[DH + 1];
          float n0 = fmaxf(pm0, m0), n1 = fmaxf(pm1, m1);
          float u0 = n0 == -INFINITY ? 0.f : n0, u1 = n1 == -INFINITY ? 0.f : n1;
          float wa0 = exp2f(pm0 - u0), wb0 = exp2f(m0 - u0), wa1 = exp2f(pm1 - u1), wb1 = exp2f(m1 - u1);
#pragma unroll
          for (int i = 0; i < DH / 8; ++i) {
            int c = i * 8 + tq * 2;
            row0[c] = row0[c] * wa0 + o[i][0] * wb0; row0[c + 1] = row0[c + 1] * wa0 + o[i][1] * wb0;
            row1[c] = row1[c] * wa1 + o[i][2] * wb1; row1[c + 1] = row1[c + 1] * wa1 + o[i][3] * wb1;
          }
          __syncwarp();
          if (tq == 0) {
            row0[DH] = n0; row0[DH + 1] = pl0 * wa0 + l0 * wb0;
            row1[DH] = n1; row1[DH + 1] = pl1 * wa1 + l1 * wb1;
          }
        }
      }
      compute_bar(NW * 32);
    }

    // ---- output: final, or partial + fixed-order merge by the last CTA of this (sequence, head) ----
    const int ct = warp * 32 + lane, nct = NW * 32;
    const float LN2 = 0.6931471805599453f;
    if (p.cluster) {
      // merged after the role branches, where every thread of the cluster meets
    } else if (p.nsplit == 1) {
      for (int idx = ct; idx < nq * DH; idx += nct) {
        int r = idx / DH, c = idx % DH;
        float l = mrg[(size_t)r * ROWF + DH + 1];
        p.out[((qrow + r) * p.H + h) * DH + c] = __float2bfloat16_rn(mrg[(size_t)r * ROWF + c] / l);
      }
      if (p.lse)
        for (int r = ct; r < nq; r += nct)
          p.lse[((size_t)b * p.H + h) * p.n + r] = (mrg[(size_t)r * ROWF + DH] + log2f(mrg[(size_t)r * ROWF + DH + 1])) * LN2;
    } else {
      float* part = p.partial + (((size_t)blockIdx.z * p.H + h) * p.nsplit) * (size_t)(NQ * ROWF);
      float* mine = part + (size_t)split * (NQ * ROWF);
      for (int idx = ct; idx < nq * ROWF; idx += nct) __stcg(mine + idx, mrg[idx]);
      __threadfence();
      compute_bar(NW * 32);
      if (ct == 0) ticket_s = atomicAdd(&p.counters[blockIdx.z * p.H + h], 1u);
      compute_bar(NW * 32);
      if (ticket_s == (unsigned)p.nsplit - 1) {
        __threadfence();
        // per-row merge weights first (one thread per row), then a wide, vectorised weighted sum
        float* wts = mrg;                                   // [nsplit][NQ], the merge buffer is free again
        for (int r = ct; r < nq; r += nct) {
          float M = -INFINITY;
          for (int s2 = 0; s2 < p.nsplit; ++s2) M = fmaxf(M, __ldcg(part + (size_t)s2 * (NQ * ROWF) + r * ROWF + DH));
          float Lsum = 0.f;
          for (int s2 = 0; s2 < p.nsplit; ++s2) {
            const float* pr = part + (size_t)s2 * (NQ * ROWF) + r * ROWF;
            float w = exp2f(__ldcg(pr + DH) - M);
            wts[s2 * NQ + r] = w;
            Lsum += __ldcg(pr + DH + 1) * w;
          }
          float inv = 1.0f / Lsum;
          for (int s2 = 0; s2 < p.nsplit; ++s2) wts[s2 * NQ + r] *= inv;
          if (p.lse) p.lse[((size_t)b * p.H + h) * p.n + r] = (M + log2f(Lsum)) * LN2;
        }
        compute_bar(NW * 32);
        constexpr int C4 = DH / 4;
        for (int idx = ct; idx < nq * C4; idx += nct) {
          const int r = idx / C4, c4 = idx % C4;
          const float4* src = reinterpret_cast<const float4*>(part + (size_t)r * ROWF) + c4;
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
          for (int s2 = 0; s2 < p.nsplit; ++s2) {
            float4 v = __ldcg(src + (size_t)s2 * (NQ * ROWF / 4));
            float w = wts[s2 * NQ + r];
            acc.x += v.x * w; acc.y += v.y * w; acc.z += v.z * w; acc.w += v.w * w;
          }
          uint2 packed = make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
          *reinterpret_cast<uint2*>(p.out + ((qrow + r) * p.H + h) * DH + c4 * 4) = packed;
        }
        if (ct == 0) p.counters[blockIdx.z * p.H + h] = 0u;       // ready for the next launch
      }
    }
  }
  if (p.cluster) {
    // The splits of this (sequence, head) are the CTAs of one cluster (rank = split): each holds its rows
    // (O, m, l) in shared memory; after the first barrier CTA r merges rows r, r + nsplit, ... from all members
    // in split order and writes the output.  Nobody leaves before the second meeting.
    cluster_start_wait();
    if (warp < NW) {
      cluster_meet(&cl_bar[0], p.nsplit, (int)threadIdx.x, wc, 303);     // every member's rows are in place
      constexpr int C4 = DH / 4;
      const int ct = warp * 32 + lane, rows_per_pass = (NW * 32) / C4;
      const float LN2 = 0.6931471805599453f;
      const uint32_t mine = smem_u32(smem_gen);
      const int c4 = ct % C4;
      for (int r = split + p.nsplit * (ct / C4); r < nq; r += p.nsplit * rows_per_pass) {
        const uint32_t row_off = (uint32_t)r * (ROWF * 4);
        float M = -INFINITY;
        for (int s2 = 0; s2 < p.nsplit; ++s2) M = fmaxf(M, ld_cluster_f32(mapa_u32(mine, (uint32_t)s2) + row_off + DH * 4));
        const float u = M == -INFINITY ? 0.f : M;
        float Lsum = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s2 = 0; s2 < p.nsplit; ++s2) {
          const uint32_t base = mapa_u32(mine, (uint32_t)s2) + row_off;
          const float w = exp2f(ld_cluster_f32(base + DH * 4) - u);
          Lsum += ld_cluster_f32(base + DH * 4 + 4) * w;
          const float4 v = ld_cluster_v4(base + (uint32_t)c4 * 16u);
          acc.x += v.x * w; acc.y += v.y * w; acc.z += v.z * w; acc.w += v.w * w;
        }
        const float inv = 1.0f / Lsum;
        *reinterpret_cast<uint2*>(p.out + ((qrow + r) * p.H + h) * DH + c4 * 4) =
            make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
        if (c4 == 0 && p.lse) p.lse[((size_t)b * p.H + h) * p.n + r] = (M + log2f(Lsum)) * LN2;
      }
      compute_bar(NW * 32);                                                          // this CTA has read all it needs
      if (warp == 0) cluster_meet_before_exit(&cl_bar[1], p.nsplit, lane, wc, &exit_flag_s, 304);
    }
    __syncthreads();                           // nobody exits before warp 0 has seen every member done
  }
}

// ---------------------------------------------------------------------------------------------
// bf16 path on the 5th-generation tensor cores (head_dim 128)
// ---------------------------------------------------------------------------------------------
// Same decomposition as above (one CTA per (split, head, sequence), 64-key tiles streamed by TMA),
// but both products run as tcgen05 MMAs with their results in tensor memory:
//   S[128 x 64]  = Q[128 x 128] . K_tile^T      (Q staged once in shared memory, zero rows past n)
//   O[128 x 128] += P[128 x 64] . V_tile        (P = p_hi + p_lo, two bf16 terms, left in tensor memory as the A operand)
// Warps 0 and 11 = TMA producers of K and V, warp 1 = TMEM allocator and QK^T issuer, warp 10 = PV issuer, warps 2-5 and 6-9 = two softmax groups
// that take alternate key tiles.  In a group thread t owns query row t (= TMEM lane t): it reads its
// whole S row from tensor memory with back-to-back loads and ONE wait (a dependent TMEM round trip
// costs ~600 cycles here, measured), keeps the running maximum and sum in registers and writes its P
// row back to tensor memory (two bf16 of neighbouring keys per column: 32 columns per term).  Each group has its own S
// buffer, its own O accumulator and its own P buffer (64 + 128 + 64 columns, twice: all 512), i.e. the two groups run two independent online-softmax streams
// over the even and the odd tiles, merged once at the end; one group's TMEM latency and arithmetic
// overlap the other's.  O stays in TMEM across tiles; it is only rescaled when a row's maximum grows
// by more than 2^8 (until then the older maximum keeps being used, which is exact after the final
// normalisation).
namespace {

constexpr uint32_t TC_KV_BYTES = 16384;               // K (or V) of one 64-key tile, two 64-wide halves
// K and V tiles travel through rings of 16 KB stages with barriers of their own: a K tile is free again as soon as its QK^T
// MMAs have retired, a V tile only after the PV MMAs one softmax later.  The depth of the rings sets the tile rate up to the
// point where the tensor pipe is busy (a freed stage is back after a TMA round trip of ~2 us): with P in shared memory (64 KB)
// there was room for two K and five V stages: 611 us at batch 16 x 128 nodes x 8K keys, 572 this way.
// (One QK^T MMA set of N = 128 over two neighbouring key tiles, filling both groups' score buffers at
// once, was tried: 24 instead of 32 MMAs per 128 keys, but the groups then run in lockstep and lose
// their overlap -- 692 against 529 us at batch 16 x 64 nodes x 8K keys.)
constexpr int TC_SK = 5, TC_SV = 6;
constexpr size_t TC_SMEM = (size_t)(TC_SK + TC_SV) * TC_KV_BYTES + 32768 + 1024;   // rings, Q, alignment slack
static_assert(TC_SMEM - 1024 >= 2 * 128 * (128 + 4) * 4, "both groups' rows fit when the key loop is over");
constexpr int TC_DH = 128, TC_ROWF = TC_DH + 4;
constexpr int TC_THREADS = 384;                       // K producer, QK^T issuer, two softmax groups of four warps, PV issuer, V producer
constexpr float TC_RESCALE = 8.0f;                    // log2 of the growth of a row maximum that forces a rescale

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) { tmem_ld16_nowait(taddr, r); }
__device__ __forceinline__ void umma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  umma_bf16(tmem_d, adesc, bdesc, idesc, acc);
}

template <bool PART>
__global__ void __launch_bounds__(TC_THREADS, 1) tree_attn_tc_kernel(const __grid_constant__ CUtensorMap tmK,
                                                                     const __grid_constant__ CUtensorMap tmV, const AttnParams p) {
  constexpr int DH = TC_DH, ROWF = TC_ROWF;
  constexpr int SK = TC_SK, SV = TC_SV;
  constexpr uint32_t QHALF = 128u * 128u, TC_Q_BYTES = 2 * QHALF;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_k[SK], empty_k[SK], full_v[SV], empty_v[SV], s_full[2], s_free[2], p_ready[2], pv_done[2], q_ready, drain_bar[2];
  __shared__ int page_list[2][kMaxPagesPerCta];               // one per producer
  __shared__ float2 ml_s[2][128];                             // a group's (m, l) of every row
  __shared__ uint32_t tmem_slot;
  __shared__ int aborted_s, exit_flag_s;
  __shared__ unsigned int ticket_s;
  __shared__ __align__(8) uint64_t cl_bar[2];
  volatile int* aborted = &aborted_s;
  const WaitCtx wc{p.wait_cycles, aborted, p.status};

  // Everything up to the first use of Q or of this step's tree keys runs before griddep_wait(): lengths,
  // live node counts and the page table were written at least two kernels ago, and so were the prefix
  // keys.  Set-up, the page list and the first prefix tiles thus overlap the previous kernel's tail.
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t q_base = smem_base;
  const uint32_t k_ring = q_base + TC_Q_BYTES;
  const uint32_t v_ring = k_ring + SK * TC_KV_BYTES;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // With one split the CTAs are persistent: (window or sequence, head) items are dealt out in turn, every second round in
  // reverse (the items come in order of falling length where they differ).  The rings run on from item to item, so that the
  // next item's first tiles arrive during this one's end.  (A CTA's beginning and end took 14 of the 25 us of an item of ten
  // tiles: batch 16 x 128 nodes x 512 keys 86 -> 62 us; the 2048-token prefill's windows 108 -> 79 us per layer.)
  const bool many = p.nsplit == 1;
  const int items = PART ? p.items : p.Bw * p.H, ctas = many ? (int)gridDim.x : 1, rounds = many ? (items + ctas - 1) / ctas : 1;
  const int split = many ? 0 : (int)blockIdx.x;
  struct Item {
    int h, b, L_old, L, nq, kv_total, t0, T, z;
    size_t qrow;
    bool too_long;
  };
  auto item_at = [&](int round) {
    Item it;
    int idx = many ? round * ctas + ((round & 1) ? ctas - 1 - (int)blockIdx.x : (int)blockIdx.x) : PART ? (int)blockIdx.y : (int)(blockIdx.z * p.H + blockIdx.y);
    it.nq = 0;
    it.T = 0;
    if (idx >= items) return it;
    if (PART) idx += p.item0;
    it.h = idx % p.H;
    it.z = idx / p.H;
    int shift;
    locate_window(p, it.z, it.b, shift);
    it.L_old = p.len[it.b];                                       // keys written by earlier launches
    it.L = it.L_old + shift;                                      // keys every row sees
    const int nq_all = (p.n_active ? min(p.n_active[it.b], p.n) : p.n) - shift;   // live nodes of this sequence (from the window on)
    it.qrow = (p.row_off ? (size_t)p.row_off[it.b] : (size_t)it.b * p.n) + shift;   // its first row of q and out
    it.nq = min(nq_all - p.row0, p.rows);                         // live query rows of this launch
    it.kv_total = it.L + min(nq_all, p.row0 + p.rows);
    const int tiles = (it.kv_total + TILE - 1) / TILE;
    const int per = (tiles + p.nsplit - 1) / p.nsplit;
    it.t0 = min(tiles, split * per);
    it.too_long = per * PAGES_PER_TILE > kMaxPagesPerCta;
    it.T = it.nq <= 0 || it.too_long ? 0 : min(tiles, it.t0 + per) - it.t0;
    return it;
  };
  if (!many && item_at(0).nq <= 0) {                              // (uniform over a cluster)
    griddep_wait();
    return;
  }
  auto enter = [&]() {                                            // (see AttnParams::follows)
    if (PART && p.follows) return;
    griddep_wait();
    griddep_launch();
  };

  if (threadIdx.x == 0) {
    aborted_s = (*p.status != 0);
    exit_flag_s = 0;
    for (int s = 0; s < SK; ++s) {
      mbar_init(smem_u32(&full_k[s]), 1);
      mbar_init(smem_u32(&empty_k[s]), 1);
    }
    for (int s = 0; s < SV; ++s) {
      mbar_init(smem_u32(&full_v[s]), 1);
      mbar_init(smem_u32(&empty_v[s]), 1);
    }
    for (int g = 0; g < 2; ++g) {
      mbar_init(smem_u32(&s_full[g]), 1);
      mbar_init(smem_u32(&s_free[g]), 4);
      mbar_init(smem_u32(&p_ready[g]), 4);
      mbar_init(smem_u32(&pv_done[g]), 1);
    }
    mbar_init(smem_u32(&q_ready), 8);
    mbar_init(smem_u32(&drain_bar[0]), 1);
    mbar_init(smem_u32(&drain_bar[1]), 1);
    mbar_init(smem_u32(&cl_bar[0]), (uint32_t)p.nsplit);
    mbar_init(smem_u32(&cl_bar[1]), (uint32_t)p.nsplit);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (p.cluster) cluster_start_arrive();
  // tensor memory: columns 0-63 / 64-127 = S of group 0 / 1, 128-255 / 256-383 = O, 384-447 / 448-511 = P (hi, lo)
  const uint32_t tmem = tmem_slot;
  float* mrg = reinterpret_cast<float*>(smem_gen);   // [2][128][ROWF] over the whole buffer, once the key loop is over

  if (warp == 0 || warp == 11) {
    // ---------------- TMA producers: warp 0 the K tiles, warp 11 the V tiles ----------------
    // A tile of K (or V) is 8 boxes of 2 KB (four pages, two 64-wide halves), issued by 8 lanes.  Issuing a box occupies its
    // warp for ~88 cycles, so one warp for both made 1400 cycles and more of every tile, the kernel's pace (572 us at batch 16 x 128 nodes x 8K keys, 465 with two).
    const bool is_v = warp == 11;
    int* list = page_list[is_v ? 1 : 0];
    const int ring = is_v ? SV : SK;
    uint64_t* full = is_v ? full_v : full_k;
    uint64_t* empty = is_v ? empty_v : empty_k;
    const uint32_t base = is_v ? v_ring : k_ring;
    static_assert(PAGES_PER_TILE == 4, "the lane -> box map below assumes four pages per tile");
    const int pg = (lane >> 1) & 3, hf = lane & 1;
    bool go = !__any_sync(0xffffffffu, *aborted), waited = false;         // a launch that starts after a time-out issues nothing
    int issued = 0, slot = 0;
    uint32_t ph = 0;
    for (int round = 0; go && round < rounds; ++round) {
      const Item it = item_at(round);
      if (it.T <= 0) continue;
      const int32_t* pt = p.page_table + (size_t)it.b * p.max_pages;
      __syncwarp();
      for (int i = lane; i < it.T * PAGES_PER_TILE; i += 32) {
        const int lp = it.t0 * PAGES_PER_TILE + i;
        list[i] = (lp * CERB_PAGE < it.kv_total && lp < p.max_pages) ? (pt[lp] * p.H + it.h) * CERB_PAGE : p.oob_row;
      }
      __syncwarp();
      for (int i = 0; i < it.T; ++i) {
        // tiles of the first ring that lie wholly inside the prefix may be fetched before the wait
        if (!waited && (issued == ring || (it.t0 + i + 1) * TILE > it.L_old)) { enter(); waited = true; }
        const uint32_t fb = smem_u32(&full[slot]);
        int stop = 0;
        if (lane == 0) {
          // (a wait that gives up says so in its return value: the consumers have stopped, nothing more is issued)
          stop = !mbar_wait_polite(smem_u32(&empty[slot]), ph ^ 1u, wc, is_v ? 306 : 305);
          if (!stop) mbar_expect_tx(fb, TC_KV_BYTES);
        }
        if (__any_sync(0xffffffffu, stop)) { go = false; break; }
        if (lane < 8) {
          const int row = list[i * PAGES_PER_TILE + pg];       // out-of-range rows are zero-filled by TMA
          tma_load_2d(base + (uint32_t)slot * TC_KV_BYTES + (uint32_t)hf * 8192u + (uint32_t)pg * (CERB_PAGE * 128), is_v ? &tmV : &tmK, hf * 64, row, fb);
        }
        ++issued;
        if (++slot == ring) { slot = 0; ph ^= 1u; }
      }
    }
    if (lane == 0 && *aborted) {
      // give-up path: the copies already issued still land in this CTA's shared memory; see each of them in
      for (int j = issued > ring ? issued - ring : 0; j < issued; ++j)
        mbar_wait_drain(smem_u32(&full[j % ring]), (uint32_t)(j / ring) & 1u, 20000000ll);
    }
    enter();             // (a lane that has waited already returns at once)
  } else if (warp == 1) {
    enter();
    // ---------------- QK^T issuer ----------------
    // (issuing one tcgen05.mma costs this thread ~95 cycles whatever its size, measured, so the two
    // products are issued by two different warps)
    {
      const uint32_t idesc_s = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);
      const uint64_t q_desc0 = desc_k_sw128(q_base), q_desc1 = desc_k_sw128(q_base + QHALF);
      bool go = !__any_sync(0xffffffffu, *aborted);
      int slot = 0, staged = 0;
      uint32_t ph = 0, used[2] = {0, 0};                 // how often each group's S buffer was written
      for (int round = 0; go && round < rounds; ++round) {
        const int T = item_at(round).T;
        if (T <= 0) continue;
        if (!mbar_wait_warp(smem_u32(&q_ready), (uint32_t)staged & 1u, wc, 308)) break;
        ++staged;
        for (int i = 0; i < T; ++i) {
          const int g = i & 1;
          if (!mbar_wait_warp(smem_u32(&full_k[slot]), ph, wc, 309) || !mbar_wait_warp(smem_u32(&s_free[g]), (used[g] & 1u) ^ 1u, wc, 311)) { go = false; break; }
          ++used[g];
          tc_fence_after();
          const uint32_t kb = k_ring + (uint32_t)slot * TC_KV_BYTES;
          const uint64_t k_desc0 = desc_k_sw128(kb), k_desc1 = desc_k_sw128(kb + 8192u);
          const uint32_t d = tmem + (uint32_t)g * 64u;
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) umma(d, q_desc0 + (uint64_t)(kk * 2), k_desc0 + (uint64_t)(kk * 2), idesc_s, kk ? 1u : 0u);
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) umma(d, q_desc1 + (uint64_t)(kk * 2), k_desc1 + (uint64_t)(kk * 2), idesc_s, 1u);
            umma_commit(smem_u32(&empty_k[slot]));     // the K tile is free once these MMAs have retired
            umma_commit(smem_u32(&s_full[g]));
          }
          __syncwarp();
          if (++slot == SK) { slot = 0; ph ^= 1u; }
        }
      }
      if (__any_sync(0xffffffffu, *aborted) && elect_one()) {                                // give-up path: see the MMAs already issued retire
        umma_commit(smem_u32(&drain_bar[0]));
        mbar_wait_drain(smem_u32(&drain_bar[0]), 0, 20000000ll);
      }
    }
  } else if (warp == 10) {
    enter();
    // ---------------- PV issuer ----------------
    {
      // B operand (V) is MN-major, N = 128 (two 64-wide swizzle atoms, p.v_lbo bytes apart)
      const uint32_t idesc_pv = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((128u >> 3) << 17) | ((128u >> 4) << 24);
      bool go = !__any_sync(0xffffffffu, *aborted);
      int slot = 0;
      uint32_t vph = 0, used[2] = {0, 0};
      for (int round = 0; go && round < rounds; ++round) {
        const int T = item_at(round).T;
        for (int j = 0; j < T; ++j) {
          const int g = j & 1;
          if (!mbar_wait_warp(smem_u32(&p_ready[g]), used[g] & 1u, wc, 312) || !mbar_wait_warp(smem_u32(&full_v[slot]), vph, wc, 313)) { go = false; break; }
          ++used[g];
          tc_fence_after();
          const uint32_t vb = v_ring + (uint32_t)slot * TC_KV_BYTES;
          const uint32_t d = tmem + 128u + (uint32_t)g * 128u;
          const uint32_t ph = tmem + 384u + (uint32_t)g * 64u, pl = ph + 32u;
          if (elect_one()) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks) {
              const uint64_t vd = desc_mn_sw128(vb + ks * 2048u, p.v_lbo, p.v_sbo);
              umma_bf16_tmem_a(d, ph + (uint32_t)(ks * 8), vd, idesc_pv, (j < 2 && ks == 0) ? 0u : 1u);
              umma_bf16_tmem_a(d, pl + (uint32_t)(ks * 8), vd, idesc_pv, 1u);
            }
            umma_commit(smem_u32(&empty_v[slot]));
            umma_commit(smem_u32(&pv_done[g]));
          }
          __syncwarp();
          if (++slot == SV) { slot = 0; vph ^= 1u; }
        }
      }
      if (__any_sync(0xffffffffu, *aborted) && elect_one()) {                                // give-up path: see the MMAs already issued retire
        umma_commit(smem_u32(&drain_bar[1]));
        mbar_wait_drain(smem_u32(&drain_bar[1]), 0, 20000000ll);
      }
    }
  } else {
    // ---------------- softmax groups: thread <-> query row, group g takes tiles g, g+2, ... ----------------
    const int g = (warp - 2) >> 2;
    const int gt = (int)threadIdx.x - 64 - g * 128;           // thread index inside the group
    const int row = (warp & 3) * 32 + lane;                    // = TMEM lane
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const int st = (int)threadIdx.x - 64;
    const float LN2 = 0.6931471805599453f;
    enter();
    int nv = 0;                                                // V tiles of the rounds before
    uint32_t n = 0;                                            // tiles this group has taken in all
    for (int round = 0; round < rounds; ++round) {
    const Item it = item_at(round);
    if (it.nq <= 0) continue;
    const int h = it.h, b = it.b, L = it.L, nq = it.nq, kv_total = it.kv_total, t0 = it.t0, T = it.T;
    const size_t qrow = it.qrow;
    const bool valid = row < nq;
    if (it.too_long && st == 0) atomicExch(p.status, CERB_E_SHAPE);
    if (T > 0) {
      // stage Q (zeros past the last node) in the swizzled K-major layout, 16-byte pieces spread over both groups
      uint4 v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int piece = st + i * 256, r = piece >> 4, c = piece & 15;
        v[i] = r < nq ? reinterpret_cast<const uint4*>(p.q + ((qrow + r) * p.H + h) * DH)[c] : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int piece = st + i * 256, r = piece >> 4, c = piece & 15;
        *reinterpret_cast<uint4*>(smem_gen + (q_base - smem_base) + (uint32_t)(c >> 3) * QHALF + (uint32_t)r * 128u +
                                  (uint32_t)(((c & 7) ^ (r & 7)) << 4)) = v[i];
      }
      proxy_fence();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&q_ready));
    }
    uint64_t anc0 = 0, anc1 = 0, anc2 = 0;
    if (valid) { anc0 = p.anc[row * CERB_ANC_WORDS]; anc1 = p.anc[row * CERB_ANC_WORDS + 1]; anc2 = p.anc[row * CERB_ANC_WORDS + 2]; }
    const uint32_t s_addr = tmem + lane_base + (uint32_t)g * 64u;
    const uint32_t o_addr = tmem + lane_base + 128u + (uint32_t)g * 128u;
    const uint32_t p_addr = tmem + lane_base + 384u + (uint32_t)g * 64u;
    float m_used = -INFINITY, l = 0.f;
    int k = 0;
    for (int i = g; i < T; i += 2, ++k, ++n) {
      mbar_wait(smem_u32(&s_full[g]), n & 1u, wc, 314);
      tc_fence_after();
      float sc[64];
#pragma unroll
      for (int c0 = 0; c0 < 64; c0 += 16) tmem_ld16(s_addr + (uint32_t)c0, reinterpret_cast<uint32_t*>(sc + c0));
      tmem_ld_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&s_free[g]));       // S is in registers: its buffer may be overwritten
      const int key0 = (t0 + i) * TILE;
      float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
      if (key0 + TILE > L) {
        const uint64_t vm = tile_visibility(key0, L, anc0, anc1, anc2);
        const uint32_t vm_lo = (uint32_t)vm, vm_hi = (uint32_t)(vm >> 32);
#pragma unroll
        for (int j = 0; j < 64; ++j) {
          const bool vis = ((j < 32 ? vm_lo >> j : vm_hi >> (j - 32)) & 1u) != 0u;      // j is a constant after unrolling
          sc[j] = vis ? sc[j] * p.scale_log2 : -INFINITY;
          mx4[j & 3] = fmaxf(mx4[j & 3], sc[j]);
        }
      } else {
#pragma unroll
        for (int j = 0; j < 64; ++j) {
          sc[j] *= p.scale_log2;
          mx4[j & 3] = fmaxf(mx4[j & 3], sc[j]);
        }
      }
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      float alpha = 1.0f;
      bool rescale = false;
      if (m_used == -INFINITY) m_used = mx;                                   // nothing accumulated for this row yet
      else if (mx > m_used + TC_RESCALE) { alpha = ex2(m_used - mx); m_used = mx; rescale = true; }
      const float mu = m_used == -INFINITY ? 0.f : m_used;
      float rs4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int j = 0; j < 64; ++j) { sc[j] = ex2(sc[j] - mu); rs4[j & 3] += sc[j]; }
      l = l * alpha + ((rs4[0] + rs4[1]) + (rs4[2] + rs4[3]));
      if (k > 0) {
        mbar_wait(smem_u32(&pv_done[g]), (n - 1u) & 1u, wc, 315);   // P buffers free, O at rest
        tc_fence_after();
        if (__any_sync(0xffffffffu, rescale)) {
#pragma unroll 1
          for (int c0 = 0; c0 < DH; c0 += 32) {
            uint32_t r[32];
            tmem_ld16(o_addr + (uint32_t)c0, r);
            tmem_ld16(o_addr + (uint32_t)c0 + 16u, r + 16);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) * alpha);
            tmem_st16(o_addr + (uint32_t)c0, r);
            tmem_st16(o_addr + (uint32_t)c0 + 16u, r + 16);
          }
          tmem_st_wait();
        }
      }
      if (key0 + TILE > kv_total) {
        // last, partial tile: rows past the end may hold anything (stale pool memory); zero V there so
        // that a zero probability times a non-finite value cannot poison the sum.  V travels apart
        // from K, so wait until it has landed.
        const int vt = nv + i;
        mbar_wait(smem_u32(&full_v[vt % SV]), (uint32_t)(vt / SV) & 1u, wc, 316);
        const int first_bad = kv_total - key0;
        uint8_t* vgen = smem_gen + (v_ring - smem_base) + (size_t)(vt % SV) * TC_KV_BYTES;
        for (int idx = gt; idx < (TILE - first_bad) * 16; idx += 128) {
          const int r = first_bad + (idx >> 4), c = idx & 15;
          *reinterpret_cast<uint4*>(vgen + (size_t)(c >> 3) * 8192 + r * 128 + (c & 7) * 16) = make_uint4(0, 0, 0, 0);
        }
      }
      // probabilities as two bf16 terms, two keys per column
#pragma unroll
      for (int c0 = 0; c0 < 32; c0 += 16) {
        uint32_t hi[16], lo[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const float p0 = sc[2 * (c0 + e)], p1 = sc[2 * (c0 + e) + 1];
          __nv_bfloat162 hb = __floats2bfloat162_rn(p0, p1);
          float2 hf = __bfloat1622float2(hb);
          hi[e] = *reinterpret_cast<uint32_t*>(&hb);
          lo[e] = pack_bf16(p0 - hf.x, p1 - hf.y);
        }
        tmem_st16(p_addr + (uint32_t)c0, hi);
        tmem_st16(p_addr + 32u + (uint32_t)c0, lo);
      }
      tmem_st_wait();
      if (key0 + TILE > kv_total) proxy_fence();      // (the zeroed rows of V)
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&p_ready[g]));
    }
    nv += T;
    if (k > 0) {
      mbar_wait(smem_u32(&pv_done[g]), (n - 1u) & 1u, wc, 317);
      tc_fence_after();
    }
    if (many) {
      // ---- output: a row's thread of group g finishes columns 64 g .. 64 g + 63 from both groups' accumulators ----
      ml_s[g][row] = make_float2(m_used, l);
      tc_fence_before();
      compute_bar(256);
      tc_fence_after();
      const float2 x0 = ml_s[0][row], x1 = ml_s[1][row];
      const float M = fmaxf(x0.x, x1.x), u = M == -INFINITY ? 0.f : M;
      const float w0 = ex2(x0.x - u), w1 = ex2(x1.x - u), Lsum = x0.y * w0 + x1.y * w1, inv = 1.0f / Lsum;
      const float f0 = w0 * inv, f1 = w1 * inv;
      bf16* o = p.out + ((qrow + (valid ? row : 0)) * p.H + h) * DH + g * 64;
      const bool wide = (reinterpret_cast<uintptr_t>(p.out) & 15) == 0;      // (8-byte alignment is all that the other routes ask for)
#pragma unroll 1
      for (int c0 = 0; c0 < 64; c0 += 16) {
        uint32_t r0[16], r1[16];
        tmem_ld16(tmem + lane_base + 128u + (uint32_t)(g * 64 + c0), r0);
        tmem_ld16(tmem + lane_base + 256u + (uint32_t)(g * 64 + c0), r1);
        tmem_ld_wait();
        uint32_t w[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          float a = __uint_as_float(r0[2 * e]) * f0, c = __uint_as_float(r0[2 * e + 1]) * f0;
          if (T > 1) {                                  // (with one tile the second group has accumulated nothing)
            a += __uint_as_float(r1[2 * e]) * f1;
            c += __uint_as_float(r1[2 * e + 1]) * f1;
          }
          w[e] = pack_bf16(a, c);
        }
        if (valid && wide) {
          reinterpret_cast<uint4*>(o + c0)[0] = make_uint4(w[0], w[1], w[2], w[3]);
          reinterpret_cast<uint4*>(o + c0)[1] = make_uint4(w[4], w[5], w[6], w[7]);
        } else if (valid) {
#pragma unroll
          for (int e = 0; e < 4; ++e) reinterpret_cast<uint2*>(o + c0)[e] = make_uint2(w[2 * e], w[2 * e + 1]);
        }
      }
      if (g == 0 && valid && p.lse) p.lse[((size_t)b * p.H + h) * p.n + row] = (M + log2f(Lsum)) * LN2;
      tc_fence_before();
      compute_bar(256);                                 // Q, the accumulators and ml_s may be written again
      tc_fence_after();
      continue;
    }
    // ---- this group's (m, l, O) rows into shared memory ----
    compute_bar(256);                               // every MMA has retired: all of shared memory can be reused
    {
      float* mr = mrg + ((size_t)g * 128 + row) * ROWF;
#pragma unroll 1
      for (int c0 = 0; c0 < DH; c0 += 32) {
        uint32_t r[32];
        if (k > 0) {
          tmem_ld16(o_addr + (uint32_t)c0, r);
          tmem_ld16(o_addr + (uint32_t)c0 + 16u, r + 16);
          tmem_ld_wait();
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) r[j] = 0u;
        }
#pragma unroll
        for (int j = 0; j < 32; j += 4)
          *reinterpret_cast<float4*>(mr + c0 + j) = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                                                __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
      }
      mr[DH] = m_used;
      mr[DH + 1] = l;
    }
    tc_fence_before();
    compute_bar(256);
    if (g == 0 && !p.cluster) {
      // merge the two groups' streams, row by row, into group 0's rows
      float* ra = mrg + (size_t)row * ROWF;
      const float* rb = mrg + ((size_t)128 + row) * ROWF;
      const float ma = ra[DH], mb = rb[DH];
      const float M = fmaxf(ma, mb), u = M == -INFINITY ? 0.f : M;
      const float wa = ex2(ma - u), wb = ex2(mb - u);
#pragma unroll 4
      for (int c = 0; c < DH; c += 4) {
        float4 a = *reinterpret_cast<float4*>(ra + c);
        const float4 bb = *reinterpret_cast<const float4*>(rb + c);
        a.x = a.x * wa + bb.x * wb; a.y = a.y * wa + bb.y * wb; a.z = a.z * wa + bb.z * wb; a.w = a.w * wa + bb.w * wb;
        *reinterpret_cast<float4*>(ra + c) = a;
      }
      ra[DH] = M;
      ra[DH + 1] = ra[DH + 1] * wa + rb[DH + 1] * wb;
    }
    compute_bar(256);

    // ---- output: final, or partial + fixed-order merge by the last CTA of this (sequence, head) ----
    const int ct = threadIdx.x - 64, nct = 256, RP = p.rows_pad;
    // (with a cluster the merge follows the role branches, where every thread of the cluster meets)
    if (!p.cluster) {
      float* part = p.partial + (((size_t)it.z * p.H + h) * p.nsplit) * (size_t)(RP * ROWF);
      float* mine = part + (size_t)split * (RP * ROWF);
      for (int idx = ct; idx < nq * ROWF; idx += nct) __stcg(mine + idx, mrg[idx]);
      __threadfence();
      compute_bar(256);
      if (ct == 0) ticket_s = atomicAdd(&p.counters[it.z * p.H + h], 1u);
      compute_bar(256);
      if (ticket_s == (unsigned)p.nsplit - 1) {
        __threadfence();
        float* wts = mrg;                                   // [nsplit][RP]
        for (int r = ct; r < nq; r += nct) {
          float M = -INFINITY;
          for (int s2 = 0; s2 < p.nsplit; ++s2) M = fmaxf(M, __ldcg(part + (size_t)s2 * (RP * ROWF) + r * ROWF + DH));
          float Lsum = 0.f;
          for (int s2 = 0; s2 < p.nsplit; ++s2) {
            const float* pr = part + (size_t)s2 * (RP * ROWF) + r * ROWF;
            float w = exp2f(__ldcg(pr + DH) - M);
            wts[s2 * RP + r] = w;
            Lsum += __ldcg(pr + DH + 1) * w;
          }
          const float inv = 1.0f / Lsum;
          for (int s2 = 0; s2 < p.nsplit; ++s2) wts[s2 * RP + r] *= inv;
          if (p.lse) p.lse[((size_t)b * p.H + h) * p.n + r] = (M + log2f(Lsum)) * LN2;
        }
        compute_bar(256);
        for (int idx = ct; idx < nq * (DH / 4); idx += nct) {
          const int r = idx / (DH / 4), c4 = idx % (DH / 4);
          const float4* src = reinterpret_cast<const float4*>(part + (size_t)r * ROWF) + c4;
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
          for (int s2 = 0; s2 < p.nsplit; ++s2) {
            const float4 v = __ldcg(src + (size_t)s2 * (RP * ROWF / 4));
            const float w = wts[s2 * RP + r];
            acc.x += v.x * w; acc.y += v.y * w; acc.z += v.z * w; acc.w += v.w * w;
          }
          *reinterpret_cast<uint2*>(p.out + ((qrow + r) * p.H + h) * DH + c4 * 4) =
              make_uint2(pack_bf16(acc.x, acc.y), pack_bf16(acc.z, acc.w));
        }
        if (ct == 0) p.counters[it.z * p.H + h] = 0u;          // ready for the next launch
      }
    }
    }
  }
  if (p.cluster) {
    // The splits of this (sequence, head) are the CTAs of one cluster (rank = split).  Each holds its merged
    // rows (O, m, l) in shared memory; once all have arrived, CTA r finishes rows r, r + nsplit, ...: it reads
    // those rows from every member in split order, weighs them and writes the final output.  Nobody leaves
    // before the second meeting, so no shared memory is read after its CTA has gone.
    cluster_start_wait();
    const Item it = item_at(0);
    const int h = it.h, b = it.b, nq = it.nq;
    const size_t qrow = it.qrow;
    if (warp >= 2 && warp < 10) {
      cluster_meet(&cl_bar[0], p.nsplit, (int)threadIdx.x - 64, wc, 318);  // every member's rows are in place
      const int ct = threadIdx.x - 64;
      const float LN2 = 0.6931471805599453f;
      const uint32_t mine = smem_u32(smem_gen);
      const int c4 = ct & 31;
      for (int r = split + p.nsplit * (ct >> 5); r < nq; r += p.nsplit * 8) {
        const uint32_t row_off = (uint32_t)r * (ROWF * 4);
        // 2 * nsplit partial rows: the two softmax groups of every split, in (split, group) order
        constexpr uint32_t GROUP_OFF = 128u * ROWF * 4u;
        float M = -INFINITY;
        for (int s2 = 0; s2 < p.nsplit; ++s2) {
          const uint32_t base = mapa_u32(mine, (uint32_t)s2) + row_off + DH * 4;
          M = fmaxf(M, fmaxf(ld_cluster_f32(base), ld_cluster_f32(base + GROUP_OFF)));
        }
        const float u = M == -INFINITY ? 0.f : M;
        float Lsum = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s2 = 0; s2 < p.nsplit; ++s2) {
#pragma unroll
          for (int gg = 0; gg < 2; ++gg) {
            const uint32_t base = mapa_u32(mine, (uint32_t)s2) + row_off + (uint32_t)gg * GROUP_OFF;
            const float w = ex2(ld_cluster_f32(base + DH * 4) - u);
            Lsum += ld_cluster_f32(base + DH * 4 + 4) * w;
            const float4 v = ld_cluster_v4(base + (uint32_t)c4 * 16u);
            acc.x += v.x * w; acc.y += v.y * w; acc.z += v.z * w; acc.w += v.w * w;
          }
        }
        const float inv = 1.0f / Lsum;
        *reinterpret_cast<uint2*>(p.out + ((qrow + r) * p.H + h) * DH + c4 * 4) =
            make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
        if (c4 == 0 && p.lse) p.lse[((size_t)b * p.H + h) * p.n + r] = (M + log2f(Lsum)) * LN2;
      }
      compute_bar(256);                                                              // this CTA has read all it needs
      if (warp == 2) cluster_meet_before_exit(&cl_bar[1], p.nsplit, lane, wc, &exit_flag_s, 319);
    }
  }
  if (PART && p.follows) {
    griddep_wait();
    griddep_launch();
  }
  tc_fence_before();
  __syncthreads();                             // nobody exits before warp 2 has seen every member done
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

}  // namespace

#include "attention_kt.cuh"

// ---------------------------------------------------------------------------------------------
// bf16, one query row per sequence (auto-regressive steps)
// ---------------------------------------------------------------------------------------------
// One CTA per (split, head, sequence), a page of 16 keys to a warp at a time, both products as plain FMA: with one row there is
// nothing for the tensor cores.  What such a launch costs at a few thousand keys is its start and its end, so it has no ring,
// no barriers and little shared memory: a lane holds 16 bytes of eight keys and eight values in registers, the first page's
// from before the wait for the kernel in front.  DH / 8 lanes share a key, the 256 / DH keys of a load are separate online
// softmaxes until the end.  The splits of a (sequence, head) are a cluster and meet in the shared memory of its first CTA.
// 32 heads of 128, against the warp-MMA kernel's 16-row layout: 16 sequences of 500 / 2000 / 8192 keys 20.9 / 75 / 299 us
// (25.9 / 82 / 308), one of 16000 39.5 (42.0); a 16-layer one-node forward of the 7B shape with 1000 keys 1270 us (1413), its
// neighbours' loads no longer waiting for an SM to be divided anew between L1 and shared memory.
constexpr int ONE_WARPS = 8;
template <int DH>
__global__ void __launch_bounds__(ONE_WARPS * 32, 2) tree_attn_one_kernel(const AttnParams p, const bf16* kpool, const bf16* vpool) {
  constexpr int LPK = DH / 8, KPL = 32 / LPK, NL = CERB_PAGE / KPL;       // lanes per key, keys per load, loads per page
  __shared__ float s_o[ONE_WARPS][DH], s_m[ONE_WARPS], s_l[ONE_WARPS];
  __shared__ float c_o[8][DH], c_m[8], c_l[8];                           // first CTA of the cluster: what every split has found
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = lane / LPK, d0 = (lane % LPK) * 8;
  const int split = blockIdx.x, h = blockIdx.y, b = blockIdx.z;
  const int L = p.len[b];
  if (p.n_active && p.n_active[b] < 1) {                                 // (every CTA of the cluster does)
    griddep_wait();
    return;
  }
  const size_t row = p.row_off ? (size_t)p.row_off[b] : (size_t)b;
  if (p.nsplit > 1) cluster_start_arrive();
  const int pages = min((L + 1 + CERB_PAGE - 1) / CERB_PAGE, p.max_pages), per = (pages + p.nsplit - 1) / p.nsplit;
  const int pg1 = min(pages, (split + 1) * per);
  const int32_t* pt = p.page_table + (size_t)b * p.max_pages;
  int pg = split * per + warp;
  auto load = [&](uint4 (&r)[NL], const bf16* pool, int at) {
    const bf16* src = pool + ((size_t)pt[at] * p.H + h) * CERB_PAGE * DH + sub * DH + d0;
#pragma unroll
    for (int i = 0; i < NL; ++i)
      asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                   : "=r"(r[i].x), "=r"(r[i].y), "=r"(r[i].z), "=r"(r[i].w) : "l"(src + i * KPL * DH) : "memory");
  };
  uint4 k[NL], v[NL];
  const bool early = pg < pg1 && (pg + 1) * CERB_PAGE <= L;              // a page without this step's key
  if (early) {
    load(k, kpool, pg);
    load(v, vpool, pg);
  }
  griddep_wait();
  griddep_launch();
  if (!early && pg < pg1) {
    load(k, kpool, pg);
    load(v, vpool, pg);
  }
  auto unpack = [](const uint4& r, float* f) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      f[2 * e] = __uint_as_float(w[e] << 16);
      f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
    }
  };
  float q[8], o[8], m = -INFINITY, l = 0.f;
  const uint32_t* qw = reinterpret_cast<const uint32_t*>(p.q + (row * p.H + h) * DH + d0);      // (q: 4-byte alignment, as for any up to 16 rows)
  unpack(make_uint4(qw[0], qw[1], qw[2], qw[3]), q);
#pragma unroll
  for (int e = 0; e < 8; ++e) o[e] = 0.f;
  for (; pg < pg1; pg += ONE_WARPS) {
    float s[NL], mx = m;
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      float f[8];
      unpack(k[i], f);
      s[i] = 0.f;
#pragma unroll
      for (int e = 0; e < 8; ++e) s[i] = fmaf(q[e], f[e], s[i]);
    }
    const bool more = pg + ONE_WARPS < pg1;
    if (more) load(k, kpool, pg + ONE_WARPS);
#pragma unroll
    for (int i = 0; i < NL; ++i) {
#pragma unroll
      for (int w = 1; w < LPK; w <<= 1) s[i] += __shfl_xor_sync(0xffffffffu, s[i], w);
      s[i] *= p.scale_log2;                                              // (the exact dot product first, as in the other kernels)
      if (pg * CERB_PAGE + i * KPL + sub > L) {                          // past the end: whatever the pool holds
        s[i] = -INFINITY;
        v[i] = make_uint4(0, 0, 0, 0);
      }
      mx = fmaxf(mx, s[i]);
    }
    const float u = mx == -INFINITY ? 0.f : mx, a = exp2f(m - u);
    m = mx;
    l *= a;
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] *= a;
#pragma unroll
    for (int i = 0; i < NL; ++i) {
      const float w = exp2f(s[i] - u);
      float f[8];
      unpack(v[i], f);
      l += w;
#pragma unroll
      for (int e = 0; e < 8; ++e) o[e] = fmaf(w, f[e], o[e]);
    }
    if (more) load(v, vpool, pg + ONE_WARPS);
  }
#pragma unroll
  for (int w = LPK; w < 32; w <<= 1) {
    const float mo = __shfl_xor_sync(0xffffffffu, m, w), lo = __shfl_xor_sync(0xffffffffu, l, w), mn = fmaxf(m, mo);
    const float u = mn == -INFINITY ? 0.f : mn, wa = exp2f(m - u), wb = exp2f(mo - u);
    l = l * wa + lo * wb;
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] = o[e] * wa + __shfl_xor_sync(0xffffffffu, o[e], w) * wb;
    m = mn;
  }
  if (lane < LPK) {
#pragma unroll
    for (int e = 0; e < 8; ++e) s_o[warp][d0 + e] = o[e];
  }
  if (lane == 0) { s_m[warp] = m; s_l[warp] = l; }
  __syncthreads();
  const int c = threadIdx.x;
  // the parts of one output (its column c, the running maxima, the sums) as one
  auto merge = [&](int parts, const float* po, const float* pm, const float* pl, float& M, float& sum) {
    M = -INFINITY;
    for (int w = 0; w < parts; ++w) M = fmaxf(M, pm[w]);
    const float u = M == -INFINITY ? 0.f : M;
    float acc = 0.f;
    sum = 0.f;
    for (int w = 0; w < parts; ++w) {
      const float f = exp2f(pm[w] - u);
      sum += pl[w] * f;
      acc += po[w * DH + c] * f;
    }
    return acc;
  };
  float acc = 0.f, M = 0.f, sum = 1.f;
  if (c < DH) acc = merge(ONE_WARPS, &s_o[0][0], s_m, s_l, M, sum);
  if (p.nsplit > 1) {
    cluster_start_wait();                                                // every CTA of the cluster runs
    if (c < DH) {
      auto put = [](float* at, float x) {
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(mapa_u32(smem_u32(at), 0)), "f"(x) : "memory");
      };
      put(&c_o[split][c], acc);
      if (c == 0) { put(&c_m[split], M); put(&c_l[split], sum); }
    }
    cluster_start_arrive();
    cluster_start_wait();                                                // ... and has left its part
    if (split != 0) return;
    if (c < DH) acc = merge(p.nsplit, &c_o[0][0], c_m, c_l, M, sum);
  }
  if (c < DH) p.out[(row * p.H + h) * DH + c] = __float2bfloat16_rn(acc / sum);
  if (c == 0 && p.lse) p.lse[((size_t)b * p.H + h) * p.n] = (M + log2f(sum)) * 0.6931471805599453f;
}

// ---------------------------------------------------------------------------------------------
// fp32 path
// ---------------------------------------------------------------------------------------------
// A CTA per (node, head), whose warps take four keys each in turn.  A launch is bound by the rounds of memory latency that one
// warp goes through, hence eight warps and not four: twelve steps and the prefill of the 4-layer fp32 model over a 64-token prompt, 2857 -> 2690 us.
// In a forward (`ahead`) the lists and (TWO) the first two fours of every warp, where they are committed keys, come ahead of the dependency
// wait, and the next four is under way while one is used: verification forwards of 4 layers with 4 heads, head_dim 64 behind 64 keys / 128 behind 500,
// 16 nodes 142.9 / 346.8 -> 139.0 / 309.1 us, 64 nodes 202.6 / 480.1 -> 195.9 / 443.9; 4 x 64 nodes behind 2000 keys (1024 CTAs) 1125 -> 1076.  More CTAs
// hide each other's latency and want the registers (80 and 114, 48 and 64 with one four): 2 x 192 nodes (1536 CTAs) 592.1 / 1606 against 596.2 / 1617;
// head_dim 128, 512 CTAs (8 x 16 nodes behind 500 keys) 666 -> 651, 1024 (a prompt of 256) 714 -> 721.
constexpr int F32_TWO_CTAS = 1024;      // (of head_dim 64)
// Of the tree's keys a node sees only its ancestors: their indices are laid out in shared memory first, so that the fours are full
// (2 x 192 nodes x 4 heads behind 16 keys: 9.8 us; 37.0 with fours of neighbouring keys, 18.5 with single ones that skip).
constexpr int F32_WARPS = 8;
template <int DH, bool TWO>
__global__ void __launch_bounds__(F32_WARPS * 32) tree_attn_f32_kernel(const float* q, const float* kpool,
                                                            const float* vpool,
                                                            const int32_t* __restrict__ page_table,
                                                            const int32_t* len, const int32_t* n_active,
                                                            const uint64_t* __restrict__ anc, float* __restrict__ out,
                                                            float* __restrict__ lse, int n, int H, int max_pages,
                                                            float scale, const int32_t* row_off, int win, int ahead) {
  constexpr int E = DH / 32;
  __shared__ float s_o[F32_WARPS][DH];
  __shared__ float s_m[F32_WARPS], s_l[F32_WARPS];
  __shared__ short s_key[CERB_MAX_NODES];
  static_assert(F32_WARPS * 32 >= CERB_MAX_NODES, "a thread per tree key");
  const bool late = !TWO || !ahead;
  if (late) {
    griddep_wait();
    griddep_launch();
  }
  // (windows of 128 rows of a prefill chunk: see locate_window)
  const int i = blockIdx.x, h = blockIdx.y, b = blockIdx.z / win, shift = (blockIdx.z % win) * kAttnRowsPerLaunch;
  const int nq_all = (n_active ? min(n_active[b], n) : n) - shift;
  const int nq = win > 1 ? min(nq_all, kAttnRowsPerLaunch) : nq_all;
  if (i >= nq) {
    if (!late) griddep_wait();      // (no CTA leaves ahead of the kernel in front)
    return;
  }
  const int settled = len[b], L = settled + shift, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // the live tree keys that this node sees, in order
  uint64_t see[CERB_ANC_WORDS];
  int seen = 0, mine = -1;                             // how many there are; the place of key threadIdx.x among them
#pragma unroll
  for (int w = 0; w < CERB_ANC_WORDS; ++w) {
    const int live = nq - 64 * w;
    see[w] = live <= 0 ? 0ull : anc[i * CERB_ANC_WORDS + w] & (live >= 64 ? ~0ull : (1ull << live) - 1ull);
    if ((int)(threadIdx.x >> 6) == w && (see[w] >> (threadIdx.x & 63)) & 1ull) mine = seen + __popcll(see[w] & ((1ull << (threadIdx.x & 63)) - 1ull));
    seen += __popcll(see[w]);
  }
  if (mine >= 0) s_key[mine] = (short)threadIdx.x;
  __syncthreads();
  float qv[E], acc[E];
  const size_t qrow = (row_off ? (size_t)row_off[b] : (size_t)b * n) + shift;
  const float* qp = q + ((qrow + i) * H + h) * DH;
  float m = -INFINITY, l = 0.f;
  // Four keys at a time, whose page entries, keys and values are all requested before the first is used: one key after the
  // other was a chain of two round trips to memory and a reduction per key.
  constexpr int KEYS = 4, ROUND = F32_WARPS * KEYS;
  const int first = warp * KEYS, end = L + seen;
  auto fetch = [&](int base, float (&kv)[KEYS][E], float (&vv)[KEYS][E], bool (&sees)[KEYS]) {
    size_t off[KEYS];
#pragma unroll
    for (int u = 0; u < KEYS; ++u) {
      int kpos = base + u;
      sees[u] = kpos < end;
      if (sees[u] && kpos >= L) kpos = L + s_key[kpos - L];
      const int page = sees[u] ? page_table[(size_t)b * max_pages + kpos / CERB_PAGE] : 0;
      off[u] = (((size_t)page * H + h) * CERB_PAGE + kpos % CERB_PAGE) * DH;
    }
#pragma unroll
    for (int u = 0; u < KEYS; ++u)
#pragma unroll
      for (int e = 0; e < E; ++e) {
        kv[u][e] = sees[u] ? kpool[off[u] + lane + 32 * e] : 0.f;
        vv[u][e] = sees[u] ? vpool[off[u] + lane + 32 * e] : 0.f;
      }
  };
  auto take = [&](const float (&kv)[KEYS][E], const float (&vv)[KEYS][E], const bool (&sees)[KEYS]) {
    float s[KEYS];
#pragma unroll
    for (int u = 0; u < KEYS; ++u) {
      s[u] = 0.f;
#pragma unroll
      for (int e = 0; e < E; ++e) s[u] += qv[e] * kv[u][e];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < KEYS; ++u) s[u] += __shfl_xor_sync(0xffffffffu, s[u], o);
    float mn = m;
#pragma unroll
    for (int u = 0; u < KEYS; ++u) {
      s[u] = sees[u] ? s[u] * scale : -INFINITY;
      mn = fmaxf(mn, s[u]);
    }
    if (mn == -INFINITY) return;                         // (nothing seen so far; uniform over the warp)
    const float al = expf(m - mn);
    l *= al;
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] *= al;
#pragma unroll
    for (int u = 0; u < KEYS; ++u) {
      const float pw = expf(s[u] - mn);
      l += pw;
#pragma unroll
      for (int e = 0; e < E; ++e) acc[e] += pw * vv[u][e];
    }
    m = mn;
  };
  float ka[KEYS][E], va[KEYS][E], kb[KEYS][E], vb[KEYS][E];              // TWO: two fours in turn
  bool sa[KEYS], sb[KEYS];
  const bool early_a = !late && first + KEYS <= settled, early_b = !late && first + ROUND + KEYS <= settled;
  if (early_a) fetch(first, ka, va, sa);
  if (early_b) fetch(first + ROUND, kb, vb, sb);
  if (!late) {
    griddep_wait();
    griddep_launch();
  }
#pragma unroll
  for (int e = 0; e < E; ++e) { qv[e] = qp[lane + 32 * e]; acc[e] = 0.f; }
  if (!TWO) {
    for (int base = first; base < end; base += ROUND) { fetch(base, ka, va, sa); take(ka, va, sa); }
  } else if (!early_a) {
    fetch(first, ka, va, sa);
  }
  for (int base = first; TWO && base < end; base += 2 * ROUND) {
    if (base + ROUND < end && !(early_b && base == first)) fetch(base + ROUND, kb, vb, sb);
    take(ka, va, sa);
    if (base + ROUND >= end) break;
    if (base + 2 * ROUND < end) fetch(base + 2 * ROUND, ka, va, sa);
    take(kb, vb, sb);
  }
  for (int e = 0; e < E; ++e) s_o[warp][lane + 32 * e] = acc[e];
  if (lane == 0) { s_m[warp] = m; s_l[warp] = l; }
  __syncthreads();
  float M = s_m[0];
#pragma unroll
  for (int w = 1; w < F32_WARPS; ++w) M = fmaxf(M, s_m[w]);
  float Ls = 0.f;
  for (int w = 0; w < F32_WARPS; ++w) Ls += s_m[w] == -INFINITY ? 0.f : s_l[w] * expf(s_m[w] - M);
  for (int c = threadIdx.x; c < DH; c += F32_WARPS * 32) {
    float a = 0.f;
    for (int w = 0; w < F32_WARPS; ++w) a += s_m[w] == -INFINITY ? 0.f : s_o[w][c] * expf(s_m[w] - M);
    out[((qrow + i) * H + h) * DH + c] = a / Ls;
  }
  if (threadIdx.x == 0 && lse) lse[((size_t)b * H + h) * n + i] = M + logf(Ls);
}

// A split reads `per` tiles of 64 keys and writes an n-row fp32 partial, so wide trees get fewer,
// longer splits: at least n/8 tiles each keeps the partial traffic near one eighth of the K/V read.
int plan_nsplit(int B, int H, int n, int max_len, int target_ctas, bool one_wave = false, int max_split = kMaxSplit) {
  int tiles = (max_len + TILE - 1) / TILE;
  if (tiles < 1) tiles = 1;
  // the tensor-core kernel holds an SM by itself: its CTAs must fit in one wave, so round down for it
  int want = one_wave ? target_ctas / (B * H) : (target_ctas + B * H - 1) / (B * H);
  int min_tiles = n / 8 > 1 ? n / 8 : 1;
  if (want > tiles / min_tiles) want = tiles / min_tiles;
  if (want > max_split) want = max_split;
  if (want > tiles) want = tiles;
  if (want < 1) want = 1;
  int per = (tiles + want - 1) / want;
  if (per * PAGES_PER_TILE > kMaxPagesPerCta) return -1;       // more than 16K keys per split
  return (tiles + per - 1) / per;
}

// How many clusters of `size` CTAs of a kernel the GPU holds at once.  A cluster lives in one GPC, so this is less than the CTAs that fit divided by
// the size: of one CTA to an SM 16 clusters of eight, and fewer than 20 of seven or 24 of six.
template <auto KERNEL>
int clusters_at_once(int threads, size_t smem, int size, int per_sm) {
  static std::atomic<int> known[9];              // (per kernel; every call would store the same)
  if (size < 2 || size > 8) return 148 * per_sm / (size < 1 ? 1 : size);
  int n = known[size].load(std::memory_order_relaxed);
  if (!n) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(size);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)size;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, KERNEL, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 148 * per_sm / size;
    }
    n = n < 1 ? 1 : n;
    known[size].store(n, std::memory_order_relaxed);
  }
  return n;
}

// The most splits, `want` at most, whose clusters are all there at once (those of a second round cost a whole round: 24 heads of 4000 keys and 64
// nodes in six splits 29.8 us, in four 18.4; 48 heads of 700 keys in three 21.0, in two 12.0).
template <typename Fits>
int splits_at_once(int tiles, int want, int items, Fits fits) {
  for (int s = want; s > 1; --s) {
    const int per = (tiles + s - 1) / s, n = (tiles + per - 1) / per;
    if (n > 1 && items <= fits(n)) return n;
  }
  return 1;
}

inline int nq_pad(int n) { return n <= 16 ? 16 : n <= 32 ? 32 : n <= 64 ? 64 : 128; }

template <int DH, int WQ, int WK, int STAGES>
int launch_cfg(AttnParams p, const CUtensorMap* tmK, const CUtensorMap* tmV, int B, int max_len, cudaStream_t st) {
  const int planned = p.nsplit;
  constexpr size_t smem = (size_t)STAGES * 2 * (DH / 64) * TILE * 128 + 1024;
  static std::atomic<bool> configured{false};
  if (!configured) {
    CERB_CUDA_OK(cudaFuncSetAttribute(tree_attn_bf16_kernel<DH, WQ, WK, STAGES>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    configured = true;
  }
  if (p.cluster) {
    const int tiles = (max_len + TILE - 1) / TILE;
    p.nsplit = splits_at_once(tiles, p.nsplit, B * p.H, [&](int n) {
      return clusters_at_once<tree_attn_bf16_kernel<DH, WQ, WK, STAGES>>((WQ * WK + 1) * 32, smem, n, WQ == 1 ? 2 : 1);
    });
    // (fewer splits are longer ones)
    if ((tiles + p.nsplit - 1) / p.nsplit * PAGES_PER_TILE > kMaxPagesPerCta) p.nsplit = planned;
    p.cluster = p.nsplit > 1 ? 1 : 0;
  }
  dim3 grid(p.nsplit, p.H, B);
  if (p.cluster)
    return launch_pdl_cluster(tree_attn_bf16_kernel<DH, WQ, WK, STAGES>, grid, dim3((WQ * WK + 1) * 32), smem, st, (unsigned)p.nsplit,
                              *tmK, *tmV, p) == cudaSuccess ? CERB_OK : CERB_E_CUDA;
  if (launch_pdl(tree_attn_bf16_kernel<DH, WQ, WK, STAGES>, grid, dim3((WQ * WK + 1) * 32), smem, st, *tmK, *tmV, p) != cudaSuccess)
    return CERB_E_CUDA;
  return CERB_OK;
}

}  // namespace

size_t attn_scratch_bytes(int B, int n, int H, int Dh) {
  size_t rows = (size_t)(kTargetCtas + B * H + kMaxSplit);
  return kCounterBytes + rows * (size_t)nq_pad(n) * (size_t)(Dh + 4) * sizeof(float);
}

// With clusters the splits of a (sequence, head) merge through distributed shared memory: at most 8 of them
// (the portable cluster size).  CERB_ATTN_CLUSTER=0 keeps the merge through global partials (up to 32 splits).
static bool attn_use_cluster() {
  static const int v = getenv("CERB_ATTN_CLUSTER") ? atoi(getenv("CERB_ATTN_CLUSTER")) : 1;
  return v != 0;
}
static int attn_max_split() { return attn_use_cluster() ? 8 : kMaxSplit; }

// One launch of the bf16 kernels over query rows row0 .. row0 + rows - 1 (rows <= 128) of every sequence's tree.
// A prefill chunk: `rows` is 128 and the launch covers its windows win0 .. win0 + win - 1 of every sequence side by side.
static int launch_attn_window(cerb_ctx* c, const cerb_attn_args* a, int row0, int rows, const CUtensorMap* tmK, const CUtensorMap* tmV,
                              int32_t* status, cudaStream_t st, const int32_t* row_off, int win = 1, int win0 = 0) {
  AttnParams p;
  const int Bw = a->B * win;             // (sequence, window) pairs
  p.items = Bw * a->n_heads;
  p.item0 = p.follows = 0;
  p.B = a->B;
  p.Bw = Bw;
  p.win = win;
  p.win0 = win0;
  const size_t row_elems = (size_t)a->n_heads * a->head_dim;
  p.q = (const bf16*)a->q + (size_t)row0 * row_elems;
  p.page_table = a->page_table;
  p.len = a->len;
  p.n_active = a->n_active;
  p.anc = a->anc + (size_t)row0 * CERB_ANC_WORDS;
  p.row_off = row_off;
  p.out = (bf16*)a->out + (size_t)row0 * row_elems;
  p.lse = a->lse ? a->lse + row0 : nullptr;
  p.row0 = row0;
  p.rows = rows;
  p.counters = (unsigned int*)a->scratch;
  p.partial = (float*)((char*)a->scratch + kCounterBytes);
  p.status = status;
  p.wait_cycles = wait_cycles();
  p.n = a->n;
  p.H = a->n_heads;
  p.max_pages = a->max_pages;
  // Which kernel: windows of 65 .. 128 rows take the tcgen05 kernel whose MMAs are 128 query rows tall; 17 .. 64 rows
  // the keys-on-M kernel (below); one row the kernel of its own; up to 16 rows the warp-MMA kernel, whose 16-row layout wastes
  // no tensor work and streams at 7.0 TB/s at batch 16 x 8K keys.  Short caches and head_dim 64 stay on the
  // warp-MMA kernel too.  CERB_ATTN_TC=0 / 1 forces the warp-MMA / the query-rows-on-M tcgen05 kernel (tests).
  static const int force_tc = getenv("CERB_ATTN_TC") ? atoi(getenv("CERB_ATTN_TC")) : -1;
  const int np_ = nq_pad(rows);
  const bool auto_tc = np_ == 128;
  const bool tensor_path = a->head_dim == 128 && (force_tc < 0 ? auto_tc : force_tc != 0);
  const bool use_cluster = attn_use_cluster();
  // CTAs that fit at once: one per SM for the tensor-core kernel and for the warp-MMA layouts of 32 rows and more
  // (288 threads x 168 registers), two per SM for the 16-row layout (160 threads); the grid is planned to fit one wave
  const int resident = (tensor_path || np_ > 16) ? 148 : kTargetCtas;
  p.nsplit = plan_nsplit(Bw, a->n_heads, np_, a->max_len, resident, true, attn_max_split());
  if (p.nsplit < 1) return CERB_E_SHAPE;
  p.oob_row = a->n_pool_pages * a->n_heads * CERB_PAGE;
  p.scale_log2 = a->scale * 1.4426950408889634f;
  p.rows_pad = nq_pad(rows);
  p.cluster = (use_cluster && p.nsplit >= 2 && p.nsplit <= 8) ? 1 : 0;
  // V tile in shared memory: [half of head_dim][64 keys][128 bytes]; 8-key groups are 1024 bytes apart
  p.v_lbo = 8192u;
  p.v_sbo = 1024u;
  int np = nq_pad(rows), rc = CERB_E_SHAPE;
  // The keys-on-M tensor-core kernel (attention_kt.cuh; 128-key tiles, every MMA row in use whatever the tree's
  // width) takes the trees of 17 to 64 nodes.  Measured inside the 7B decoding step, batch 1, 2K keys, this kernel
  // against the others: 64-node steps 4.33 / 4.47 ms, one-node steps 3.39 / 3.27 ms (the 16-row warp-MMA layout has
  // less to set up); alone at batch 16 x 8K keys: 64 nodes 403 / 537 us, 16 nodes 392 / 308 us, 128 nodes (its
  // 128-query form, not built any more) 654 / 572 us.  CERB_ATTN_KT=0 / 1 keeps it off / uses it for every launch of
  // up to 64 rows (tests).
  static const int force_kt = getenv("CERB_ATTN_KT") ? atoi(getenv("CERB_ATTN_KT")) : -1;
  // One row per sequence: the kernel without tensor cores, at every length (figures there); the switches for tests keep it off.
  if (a->n == 1 && win == 1 && use_cluster && force_tc < 0 && force_kt < 0) {
    // two CTAs to an SM, at least a page to a warp
    int want = 2 * 148 / (a->B * a->n_heads);
    const int pages = (a->max_len + CERB_PAGE - 1) / CERB_PAGE;
    if (want > (pages + ONE_WARPS - 1) / ONE_WARPS) want = (pages + ONE_WARPS - 1) / ONE_WARPS;
    want = want < 1 ? 1 : want > 8 ? 8 : want;
    while (want > 1 && a->B * a->n_heads > (a->head_dim == 128 ? clusters_at_once<tree_attn_one_kernel<128>>(ONE_WARPS * 32, 0, want, 2)
                                                                : clusters_at_once<tree_attn_one_kernel<64>>(ONE_WARPS * 32, 0, want, 2)))
      --want;
    p.nsplit = want;
    auto kern = a->head_dim == 128 ? tree_attn_one_kernel<128> : tree_attn_one_kernel<64>;
    const dim3 grid(p.nsplit, p.H, Bw), block(ONE_WARPS * 32);
    const bf16 *kp = (const bf16*)a->k_pool, *vp = (const bf16*)a->v_pool;
    if (p.nsplit > 1) return launch_pdl_cluster(kern, grid, block, 0, st, (unsigned)p.nsplit, p, kp, vp) == cudaSuccess ? CERB_OK : CERB_E_CUDA;
    return launch_pdl(kern, grid, block, 0, st, p, kp, vp) == cudaSuccess ? CERB_OK : CERB_E_CUDA;
  }
  const bool kt_path = a->head_dim == 128 && force_tc < 0 && rows <= 64 && (force_kt < 0 ? rows > 16 : force_kt != 0);
  if (kt_path || tensor_path) {
    static std::atomic<bool> configured{false};
    if (!configured) {
      for (auto kern : {tree_attn_kt_kernel<false>, tree_attn_kt_kernel<true>})
        CERB_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)KT_SMEM));
      for (auto kern : {tree_attn_tc_kernel<false>, tree_attn_tc_kernel<true>})
        CERB_CUDA_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM));
      configured = true;
    }
    const int items = p.items, tile = kt_path ? KT_TILE : TILE, tiles = (a->max_len + tile - 1) / tile;
    // A launch over `n_items` of the (sequence or window, head) pairs, whose keys are cut into `nsplit` splits.  The kernels' forms for a part of
    // the items or for a launch that follows are instances of their own: with the tests in the others these took 0.6 us more.
    auto launch = [&](int n_items, int nsplit) {
      p.items = n_items;
      p.nsplit = nsplit;
      p.cluster = (use_cluster && nsplit >= 2 && nsplit <= 8) ? 1 : 0;
      const bool part = n_items != items || p.follows;
      auto go = [&](auto kern, dim3 grid, int threads, size_t smem) {
        return (p.cluster ? launch_pdl_cluster(kern, grid, dim3(threads), smem, st, (unsigned)nsplit, *tmK, *tmV, p)
                          : launch_pdl(kern, grid, dim3(threads), smem, st, *tmK, *tmV, p)) == cudaSuccess ? CERB_OK : CERB_E_CUDA;
      };
      const dim3 grid = part ? dim3(nsplit, n_items) : dim3(nsplit, p.H, Bw);
      if (kt_path) return go(part ? tree_attn_kt_kernel<true> : tree_attn_kt_kernel<false>, grid, KT_THREADS, KT_SMEM);
      // one split: persistent CTAs over the items
      return go(part ? tree_attn_tc_kernel<true> : tree_attn_tc_kernel<false>, nsplit == 1 ? dim3(n_items < 148 ? n_items : 148) : grid, TC_THREADS, TC_SMEM);
    };
    auto splits = [&](int n_items) {
      int planned;
      if (kt_path) {
        int want = 148 / n_items;
        if (want > attn_max_split()) want = attn_max_split();
        if (want > tiles) want = tiles;
        if (want < 1) want = 1;
        const int per = (tiles + want - 1) / want;
        planned = (tiles + per - 1) / per;
      } else {
        planned = plan_nsplit(n_items, 1, np_, a->max_len, resident, true, attn_max_split());
      }
      int ns = planned;
      if (use_cluster && ns > 1)
        ns = splits_at_once(tiles, ns, n_items, [&](int n) {
          return kt_path ? clusters_at_once<tree_attn_kt_kernel<false>>(KT_THREADS, KT_SMEM, n, 1) : clusters_at_once<tree_attn_tc_kernel<false>>(TC_THREADS, TC_SMEM, n, 1);
        });
      // A launch that follows runs on the SMs that the first one leaves, and its clusters have to find room there: in 104 CTAs at most, as long as a split is no longer
      // than eight tiles.  (150 nodes, 24 items of 1000 keys in five splits 32.2 us, in three 24.0, without following 30.9; 36 of 600 28.6, 19.7, 27.9; 32 of 3000 keys,
      // four splits and three of nine tiles: 45.4, 46.6, 46.2.)
      if (p.follows) {
        int m = ns;
        while (m > 1 && n_items * m > 104) {
          const int per = (tiles + m - 2) / (m - 1);
          m = (tiles + per - 1) / per;
        }
        if ((tiles + m - 1) / m <= 8) ns = m;
      }
      const int pages = kt_path ? KT_PAGES : PAGES_PER_TILE;
      auto too_long = [&](int n) { return (tiles + n - 1) / n * pages > kMaxPagesPerCta; };      // (fewer splits are longer ones)
      if (ns > 0 && too_long(ns)) ns = planned;
      return ns < 1 || too_long(ns) ? -1 : ns;
    };
    p.follows = row0 > 0 && use_cluster ? 1 : 0;                     // the second window of a wide tree (150 nodes behind 600 keys 28.4 -> 20.2 us)
    // More items than SMs: where the last round leaves half of the SMs and more without one, its items' keys are split over them in a launch of its
    // own, which needs nothing from the first one.  160 heads of 800 / 1564 / 4096 keys, 64 nodes: 30.7 / 44.9 / 94.9 us in one launch, 26.9 / 35.9 / 65.4 in two;
    // 512: 65.6 / 95.4 / 217 and 66.1 / 91.8 / 201; below 768 keys the second launch costs as much as it gives (300 keys: 0.88 to 0.97 x), and with a rest of more than 24,
    // whose keys are cut into few splits, below 1024 (24 nodes behind 740 keys, 352 / 480 / 512 / 640 items: 0.99 / 0.99 / 0.975 / 0.96 x).
    const int rest = items % 148;
    if (win == 1 && use_cluster && items > 148 && rest > 0 && rest <= 74 && tiles * tile >= (rest <= 24 ? 768 : 1024)) {
      const int ns = splits(rest);
      if (ns > 1 && splits(items) == 1) {
        rc = launch(items - rest, 1);
        if (rc != CERB_OK) return rc;
        CERB_LAUNCH_CHECK(c);
        p.item0 = items - rest;
        p.follows = 1;
        return launch(rest, ns);
      }
    }
    const int ns = splits(items);
    if (ns < 1) return CERB_E_SHAPE;
    rc = launch(items, ns);
  } else if (a->head_dim == 128) {
    if (np == 16) rc = launch_cfg<128, 1, 4, 3>(p, tmK, tmV, Bw, a->max_len, st);
    else if (np == 32) rc = launch_cfg<128, 2, 4, 3>(p, tmK, tmV, Bw, a->max_len, st);
    else if (np == 64) rc = launch_cfg<128, 4, 2, 3>(p, tmK, tmV, Bw, a->max_len, st);
    else rc = launch_cfg<128, 8, 1, 3>(p, tmK, tmV, Bw, a->max_len, st);
  } else if (a->head_dim == 64) {
    if (np == 16) rc = launch_cfg<64, 1, 4, 4>(p, tmK, tmV, Bw, a->max_len, st);
    else if (np == 32) rc = launch_cfg<64, 2, 4, 4>(p, tmK, tmV, Bw, a->max_len, st);
    else if (np == 64) rc = launch_cfg<64, 4, 2, 4>(p, tmK, tmV, Bw, a->max_len, st);
    else rc = launch_cfg<64, 8, 1, 4>(p, tmK, tmV, Bw, a->max_len, st);
  }
  return rc;
}

int launch_tree_attention(cerb_ctx* c, const cerb_attn_args* a, const CUtensorMap* tmK, const CUtensorMap* tmV,
                          int sm_count, int32_t* status, cudaStream_t st, const int32_t* row_off, bool chain) {
  (void)sm_count;
  const int win = chain ? (a->n + kAttnRowsPerLaunch - 1) / kAttnRowsPerLaunch : 1;
  if (a->dtype == CERB_F32) {
    dim3 grid(win > 1 ? kAttnRowsPerLaunch : a->n, a->n_heads, a->B * win);
    const bool two = (long long)grid.x * grid.y * grid.z * a->head_dim <= F32_TWO_CTAS * 64;
    auto go = [&](auto kern) {
      launch_pdl(kern, grid, dim3(F32_WARPS * 32), 0, st, (const float*)a->q, (const float*)a->k_pool, (const float*)a->v_pool, a->page_table, a->len,
                 a->n_active, a->anc, (float*)a->out, a->lse, a->n, a->n_heads, a->max_pages, a->scale, row_off, win, c && two ? 1 : 0);
    };
    if (a->head_dim == 64)
      two ? go(tree_attn_f32_kernel<64, true>) : go(tree_attn_f32_kernel<64, false>);
    else if (a->head_dim == 128)
      two ? go(tree_attn_f32_kernel<128, true>) : go(tree_attn_f32_kernel<128, false>);
    else
      return CERB_E_SHAPE;
    CERB_LAUNCH_CHECK(c);
    return CERB_OK;
  }
  if (a->B * a->n_heads > (int)(kCounterBytes / sizeof(unsigned int)) - 4) return CERB_E_SHAPE;   // last 16 bytes: status word
  if (win > 1) {
    // a prefill chunk of more than 128 tokens per sequence: its windows are CTAs of one launch
    if (a->scratch_bytes < attn_scratch_bytes(a->B, kAttnRowsPerLaunch, a->n_heads, a->head_dim)) return CERB_E_NOMEM;
    // ... of as few as there is a plan for: with many windows no keys are split, and a CTA's page list ends at 16384 keys
    int per = win;
    while (per > 1 && plan_nsplit(a->B * per, a->n_heads, kAttnRowsPerLaunch, a->max_len, 148, true, attn_max_split()) < 1) --per;
    const int launches = (win + per - 1) / per;
    per = (win + launches - 1) / launches;
    for (int win0 = 0; win0 < win; win0 += per) {
      CERB_TRY(launch_attn_window(c, a, 0, kAttnRowsPerLaunch, tmK, tmV, status, st, row_off, win - win0 < per ? win - win0 : per, win0));
      CERB_LAUNCH_CHECK(c);
    }
    return CERB_OK;
  }
  if (a->scratch_bytes < attn_scratch_bytes(a->B, a->n, a->n_heads, a->head_dim)) return CERB_E_NOMEM;
  // A CTA holds at most 128 query rows (the tensor-core MMA's height, eight 16-row warps in the warp-MMA kernel).
  // A wider tree (Sec. 5.1 goes up to 150 candidates + the root) takes one launch per window of 128 rows; the
  // launches are stream-ordered and share the scratch.  Keys are not windowed: rows of the second window see the
  // whole tree, rows of the first only nodes below 128 (an ancestor has a lower index than its descendant).
  for (int row0 = 0; row0 < a->n; row0 += kAttnRowsPerLaunch) {
    const int rows = a->n - row0 < kAttnRowsPerLaunch ? a->n - row0 : kAttnRowsPerLaunch;
    CERB_TRY(launch_attn_window(c, a, row0, rows, tmK, tmV, status, st, row_off));
    CERB_LAUNCH_CHECK(c);
  }
  return CERB_OK;
}

}  // namespace cerb

// ---------------------------------------------------------------------------------------------
// Tree attention for callers that cannot allocate device memory
// ---------------------------------------------------------------------------------------------
// The split-KV partials and ticket counters normally live in a scratch buffer the caller allocates.
// Some callers cannot do that: code running inside a memory-pool or allocator callback, a plug-in
// that is handed fixed buffers by its host application, or a process whose device-memory budget was
// fixed at start-up.  For them the scratch lives in this library's image instead, as one static
// device array.  Every GPU that loads the library holds these bytes until the process exits.
static __device__ __align__(256) unsigned char g_static_attn_scratch[CERB_STATIC_ATTN_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::atomic<void*> g_static_scratch_addr[kMaxDevices];      // device address of the array, per device, once known

// Set-up, once per device, with that device current.  In host code the array's name is only a handle; the
// address a kernel can use has to be asked for.  Two threads racing here both get the same answer from the
// runtime, so the slot is simply an atomic pointer.
int static_scratch(void** out) {
  int dev = -1;
  CERB_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return CERB_E_SHAPE;
  void* ptr = g_static_scratch_addr[dev].load(std::memory_order_acquire);
  if (!ptr) {
    if (cudaGetSymbolAddress(&ptr, g_static_attn_scratch) != cudaSuccess || !ptr) return CERB_E_CUDA;
    g_static_scratch_addr[dev].store(ptr, std::memory_order_release);
  }
  *out = ptr;
  return CERB_OK;
}
}  // namespace

extern "C" int cerb_tree_attention_noalloc(const cerb_attn_args* a, void* stream) {
  using namespace cerb;
  if (!a || !a->q || !a->k_pool || !a->v_pool || !a->page_table || !a->len || !a->anc || !a->out) return CERB_E_ARG;
  if (a->B < 1 || a->n < 1 || a->n > CERB_MAX_NODES || a->n_heads < 1 || a->n_pool_pages < 1) return CERB_E_ARG;
  if (a->dtype != CERB_BF16) return CERB_E_ARG;
  if (a->head_dim != 64 && a->head_dim != 128) return CERB_E_SHAPE;
  const size_t need = attn_scratch_bytes(a->B, a->n, a->n_heads, a->head_dim);
  if (need > (size_t)CERB_STATIC_ATTN_SCRATCH_BYTES) return CERB_E_NOMEM;     // problem too large for the built-in scratch
  void* scratch = nullptr;
  CERB_TRY(static_scratch(&scratch));
  cudaStream_t st = (cudaStream_t)stream;
  // The array keeps whatever the previous call left.  The ticket counters must start at zero; the partials behind
  // them are fully rewritten before being read.  The status words (the last 16 bytes of the first 4 KB) are NOT
  // cleared here: a time-out stays visible until cerb_tree_attention_noalloc_status has read it.
  CERB_CUDA_OK(cudaMemsetAsync(scratch, 0, kCounterBytes - 16, st));
  CUtensorMap tk, tv;
  CERB_TRY(make_pool_map(&tk, a->k_pool, a->n_pool_pages, a->n_heads, a->head_dim));
  CERB_TRY(make_pool_map(&tv, a->v_pool, a->n_pool_pages, a->n_heads, a->head_dim));
  cerb_attn_args b = *a;
  b.scratch = scratch;
  b.scratch_bytes = CERB_STATIC_ATTN_SCRATCH_BYTES;
  int32_t* status = reinterpret_cast<int32_t*>((char*)scratch + kCounterBytes - 16);
  return launch_tree_attention(nullptr, &b, &tk, &tv, 148, status, st);
}

extern "C" int cerb_tree_attention_noalloc_status(void* stream) {
  using namespace cerb;
  void* scratch = nullptr;
  CERB_TRY(static_scratch(&scratch));
  CERB_CUDA_OK(cudaStreamSynchronize((cudaStream_t)stream));
  int32_t words[4] = {0, 0, 0, 0};
  CERB_CUDA_OK(cudaMemcpy(words, (char*)scratch + kCounterBytes - 16, sizeof(words), cudaMemcpyDeviceToHost));
  if (words[0] != 0) CERB_CUDA_OK(cudaMemset((char*)scratch + kCounterBytes - 16, 0, 16));
  return words[0];
}
