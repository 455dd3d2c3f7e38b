// Entropy gate (Section 4.2) and greedy acceptance with KV compaction (Section 3.1).
#include "cerb_internal.cuh"

namespace cerb {

namespace {

template <typename T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ldf<bf16>(const bf16* p) { return __bfloat162float(*p); }

__device__ __forceinline__ float block_reduce(float v, float* red, bool is_max) {
  for (int o = 16; o > 0; o >>= 1) {
    float t = __shfl_xor_sync(0xffffffffu, v, o);
    v = is_max ? fmaxf(v, t) : v + t;
  }
  int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  float r = red[0];
  for (int i = 1; i < nw; ++i) r = is_max ? fmaxf(r, red[i]) : r + red[i];
  return r;
}

// P = Softmax(h_last) over the d_model components; S = -sum P log2 P.
// With m = max h, Z = sum e^(h-m), A = sum e^(h-m) (h-m):  S = (ln Z - A / Z) / ln 2.
// mode = S > T ? auto-regressive : parallel (Algorithm 1).
template <typename T>
__global__ void __launch_bounds__(256) gate_kernel(const T* h_last, int d, float thr, float* __restrict__ S,
                                                   int32_t* __restrict__ mode, int32_t* __restrict__ n_active, int n_par,
                                                   const int32_t* len, int32_t* __restrict__ host) {
  __shared__ float red[32];
  griddep_wait();
  griddep_launch();
  const T* h = h_last + (size_t)blockIdx.x * d;
  float m = -INFINITY;
  for (int j = threadIdx.x; j < d; j += blockDim.x) m = fmaxf(m, ldf(h + j));
  m = block_reduce(m, red, true);
  float z = 0.f, a = 0.f;
  for (int j = threadIdx.x; j < d; j += blockDim.x) {
    float t = ldf(h + j) - m, e = expf(t);
    z += e;
    a += e * t;
  }
  // (both sums in one go; the order of each is that of block_reduce)
  for (int o = 16; o > 0; o >>= 1) {
    z += __shfl_xor_sync(0xffffffffu, z, o);
    a += __shfl_xor_sync(0xffffffffu, a, o);
  }
  __shared__ float2 both[32];
  if ((threadIdx.x & 31) == 0) both[threadIdx.x >> 5] = make_float2(z, a);
  __syncthreads();
  if (threadIdx.x == 0) {
    z = both[0].x;
    a = both[0].y;
    for (int i = 1; i < (int)blockDim.x >> 5; ++i) { z += both[i].x; a += both[i].y; }
    float s = (logf(z) - a / z) * 1.4426950408889634f;
    int md = s > thr ? CERB_MODE_AR : CERB_MODE_PAR;
    S[blockIdx.x] = s;
    mode[blockIdx.x] = md;
    if (n_active) n_active[blockIdx.x] = md == CERB_MODE_AR ? 1 : n_par;
    if (host) {
      // the step's one read-back, written to pinned host memory here: mode, length and S
      host[blockIdx.x] = md;
      host[CERB_MAX_BATCH + blockIdx.x] = len[blockIdx.x];
      host[2 * CERB_MAX_BATCH + blockIdx.x] = __float_as_int(s);
      __threadfence_system();
    }
  }
}

// One CTA of 192 threads (CERB_MAX_NODES) per sequence, thread v <-> node v.
//   match[v] = token of v equals the model's argmax at v's parent   (root: always)
//   v is accepted-reachable iff every node on its root path matches: (anc[v] & ~match) == 0
//   winner = deepest reachable node, lowest index among equals; its ancestors, ascending, are the path.
// What the host reads goes straight to its pinned memory (host_n, host_tok, where the caller's is pinned): two copies of a few words behind
// the step took 2.7 us each, and the next step's gate could not start while the compaction drains.  Twelve steps and the prefill of the 4-layer
// fp32 model 1905 -> 1780 us, 48 steps of the 7B shape 1.027 -> 1.040 x the build without.
template <typename T>
__global__ void __launch_bounds__(CERB_MAX_NODES) accept_kernel(const int32_t* tok, const int32_t* argmax, const int32_t* n_active,
                                                     const int32_t* __restrict__ parent, const int32_t* __restrict__ depth,
                                                     const uint64_t* __restrict__ anc, int n, int32_t* len,
                                                     int32_t* __restrict__ len_old, int32_t* __restrict__ root,
                                                     const T* hidden, T* __restrict__ h_last, int d,
                                                     int32_t* __restrict__ n_accept, int32_t* __restrict__ path,
                                                     int32_t* __restrict__ out_tok, const int32_t* row_off,
                                                     int32_t* __restrict__ host_n, int32_t* __restrict__ host_tok) {
  constexpr int NWARP = CERB_MAX_NODES / 32;
  __shared__ uint32_t mword[NWARP];
  __shared__ int skey[NWARP];
  __shared__ int best_s;
  __shared__ int tok_s[CERB_MAX_NODES], am_s[CERB_MAX_NODES];
  const int b = blockIdx.x, v = threadIdx.x;
  // ahead of the wait: the tree.  The lengths are not: of two calls for trees of one node the second follows the kernel that writes them.
  const size_t row0 = row_off ? (size_t)row_off[b] : (size_t)b * n;      // this sequence's first row of argmax / hidden
  const int at = v < n ? v : 0;
  const int up = at ? parent[at] : 0, level = depth[at];
  uint64_t see[CERB_ANC_WORDS];
#pragma unroll
  for (int w = 0; w < CERB_ANC_WORDS; ++w) see[w] = anc[at * CERB_ANC_WORDS + w];
  griddep_wait();
  griddep_launch();
  // (all of these on their way together; the rows of nodes that are not live lie inside the buffers)
  const int na = min(n_active[b], n), mine = tok[(size_t)b * n + at], above = argmax[row0 + up], own = argmax[row0 + at], L = len[b];
  tok_s[v] = mine;
  am_s[v] = own;
  bool match = v < na && (v == 0 || mine == above);
  uint32_t bal = __ballot_sync(0xffffffffu, match);
  if ((v & 31) == 0) mword[v >> 5] = bal;
  __syncthreads();
  uint64_t mm[CERB_ANC_WORDS];
#pragma unroll
  for (int w = 0; w < CERB_ANC_WORDS; ++w) mm[w] = (uint64_t)mword[2 * w] | ((uint64_t)mword[2 * w + 1] << 32);
  int key = -1;
  if (v < na) {
    bool reach = true;
#pragma unroll
    for (int w = 0; w < CERB_ANC_WORDS; ++w) reach = reach && (see[w] & ~mm[w]) == 0;
    if (reach) key = level * 256 + (255 - v);
  }
  for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
  if ((v & 31) == 0) skey[v >> 5] = key;
  __syncthreads();
  int k = skey[0];
#pragma unroll
  for (int w = 1; w < NWARP; ++w) k = max(k, skey[w]);
  const int best = k < 0 ? 0 : 255 - (k & 255);
  if (v == best) {
    best_s = best;
    int cnt = 0;
#pragma unroll
    for (int w = 0; w < CERB_ANC_WORDS; ++w) {
      uint64_t bits = see[w];
      while (bits && cnt < kPathMax) {
        int j = __ffsll((long long)bits) - 1;
        bits &= bits - 1;
        path[(size_t)b * kPathMax + cnt] = w * 64 + j;
        out_tok[(size_t)b * kPathMax + cnt] = tok_s[w * 64 + j];
        if (host_tok) host_tok[(size_t)b * kPathMax + cnt] = tok_s[w * 64 + j];
        ++cnt;
      }
    }
    for (int j = cnt; j < kPathMax; ++j) {
      path[(size_t)b * kPathMax + j] = -1;
      out_tok[(size_t)b * kPathMax + j] = -1;
      if (host_tok) host_tok[(size_t)b * kPathMax + j] = -1;
    }
    n_accept[b] = cnt;
    if (host_n) host_n[b] = cnt;
    root[b] = am_s[best];
    len_old[b] = L;
    len[b] = L + cnt;
  }
  __syncthreads();
  const T* src = hidden + (row0 + best_s) * d;
  for (int j = threadIdx.x; j < d; j += blockDim.x) h_last[(size_t)b * d + j] = src[j];
}

// Move the accepted nodes' K/V from slot L + path[j] to slot L + j in every layer.  One thread owns
// one 16-byte column chunk of one (layer, K|V, head) and loads all path rows before storing any:
// path[j] >= j, so a destination may be a later source.
__global__ void kv_compact_kernel(char* kpool, char* vpool, size_t layer_bytes,
                                  const int32_t* __restrict__ page_table, int max_pages,
                                  const int32_t* len_old, const int32_t* n_accept, const int32_t* path, int H, int row_bytes) {
  griddep_wait();
  griddep_launch();
  const int b = blockIdx.z, layer = blockIdx.y >> 1;
  char* pool = ((blockIdx.y & 1) ? vpool : kpool) + (size_t)layer * layer_bytes;
  const int chunks = row_bytes / 16;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= H * chunks) return;
  const int h = idx / chunks, ch = idx % chunks;
  const int cnt = n_accept[b], L = len_old[b];
  const int32_t* pt = page_table + (size_t)b * max_pages;
  uint4 regs[kPathMax];
  bool moved[kPathMax];
#pragma unroll
  for (int j = 0; j < kPathMax; ++j) {
    moved[j] = false;
    if (j < cnt) {
      int pj = path[(size_t)b * kPathMax + j];
      if (pj != j) {
        int slot = L + pj;
        size_t off = (((size_t)pt[slot / CERB_PAGE] * H + h) * CERB_PAGE + slot % CERB_PAGE) * row_bytes + (size_t)ch * 16;
        regs[j] = *reinterpret_cast<const uint4*>(pool + off);
        moved[j] = true;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < kPathMax; ++j) {
    if (moved[j]) {
      int slot = L + j;
      size_t off = (((size_t)pt[slot / CERB_PAGE] * H + h) * CERB_PAGE + slot % CERB_PAGE) * row_bytes + (size_t)ch * 16;
      *reinterpret_cast<uint4*>(pool + off) = regs[j];
    }
  }
}

}  // namespace

// (Like every kernel of a step, these start while the kernel in front drains: together with the fp32 attention's launches 2689
// -> 2557 us for twelve steps and the prefill of the 4-layer fp32 model.)
int launch_gate(cerb_ctx* c, float T, float* S, int32_t* mode, int32_t* nactive_or_null, int n_par, cudaStream_t st, int32_t* host) {
  int d = c->cfg.d_model;
  if (c->bf16) launch_pdl(gate_kernel<bf16>, dim3(c->B), dim3(256), 0, st, (const bf16*)c->d_hlast, d, T, S, mode, nactive_or_null, n_par, (const int32_t*)c->d_len, host);
  else launch_pdl(gate_kernel<float>, dim3(c->B), dim3(256), 0, st, (const float*)c->d_hlast, d, T, S, mode, nactive_or_null, n_par, (const int32_t*)c->d_len, host);
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

int launch_accept(cerb_ctx* c, const cerb_tree* tree, const int32_t* tree_tok, const int32_t* n_active,
                  const int32_t* node_argmax, int32_t* n_accept, int32_t* path, int32_t* out_tok, cudaStream_t st,
                  const int32_t* row_off, int32_t* host_n, int32_t* host_tok) {
  const cerb_config& g = c->cfg;
  const TreeDev& t = tree->dev;
  if (c->bf16)
    launch_pdl(accept_kernel<bf16>, dim3(c->B), dim3(CERB_MAX_NODES), 0, st, tree_tok, node_argmax, n_active, (const int32_t*)t.parent,
               (const int32_t*)t.depth, (const uint64_t*)t.anc, tree->n, c->d_len, c->d_len_old, c->d_root, (const bf16*)c->d_hidden,
               (bf16*)c->d_hlast, g.d_model, n_accept, path, out_tok, row_off, host_n, host_tok);
  else
    launch_pdl(accept_kernel<float>, dim3(c->B), dim3(CERB_MAX_NODES), 0, st, tree_tok, node_argmax, n_active, (const int32_t*)t.parent,
               (const int32_t*)t.depth, (const uint64_t*)t.anc, tree->n, c->d_len, c->d_len_old, c->d_root, (const float*)c->d_hidden,
               (float*)c->d_hlast, g.d_model, n_accept, path, out_tok, row_off, host_n, host_tok);
  CERB_LAUNCH_CHECK(c);
  if (tree->n > 1) {
    int row_bytes = g.head_dim * (int)c->esize;
    int threads = g.n_heads * (row_bytes / 16);
    dim3 grid((threads + 127) / 128, g.n_layers * 2, c->B);
    launch_pdl(kv_compact_kernel, grid, dim3(128), 0, st, (char*)c->k_pool, (char*)c->v_pool, c->pool_layer_bytes, c->page_table, g.max_pages,
               (const int32_t*)c->d_len_old, (const int32_t*)n_accept, (const int32_t*)path, g.n_heads, row_bytes);
    CERB_LAUNCH_CHECK(c);
  }
  return CERB_OK;
}

}  // namespace cerb
