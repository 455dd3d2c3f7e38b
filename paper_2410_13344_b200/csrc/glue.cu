// Small element-wise kernels of the base-model forward (Algorithm 1: embedding, TL_i, LH):
// embedding gather, RMSNorm, RoPE + KV-page append, residual add, SwiGLU, row argmax.
// GEMM outputs arrive as fp32 split-K partial sums [split][row][col]; every consumer here
// adds the splits in index order, so results do not depend on scheduling.
#include <type_traits>

#include "cerb_internal.cuh"

namespace cerb {

template <typename T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ldf<bf16>(const bf16* p) { return __bfloat162float(*p); }
template <typename T> __device__ __forceinline__ void stf(T* p, float v);
template <> __device__ __forceinline__ void stf<float>(float* p, float v) { *p = v; }
template <> __device__ __forceinline__ void stf<bf16>(bf16* p, float v) { *p = __float2bfloat16_rn(v); }

__device__ __forceinline__ float block_sum(float v, float* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  float t = 0.f;
  for (int i = 0; i < nw; ++i) t += red[i];
  return t;
}


// cos/sin of pos * base^(-2i/Dh), evaluated once in double precision.
__global__ void rope_table_kernel(float2* tab, int max_pos, int half, double base) {
  int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= max_pos * half) return;
  int pos = idx / half, i = idx % half;
  double inv = pow(base, -2.0 * (double)i / (double)(2 * half));
  double s, c;
  sincos((double)pos * inv, &s, &c);
  tab[idx] = make_float2((float)c, (float)s);
}

template <typename T> __device__ __forceinline__ void ld4(const T* p, float* f);
template <> __device__ __forceinline__ void ld4<float>(const float* p, float* f) {
  float4 v = *reinterpret_cast<const float4*>(p);
  f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
template <> __device__ __forceinline__ void ld4<bf16>(const bf16* p, float* f) {
  uint2 v = *reinterpret_cast<const uint2*>(p);
  float2 a = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&v.x)), b = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162*>(&v.y));
  f[0] = a.x; f[1] = a.y; f[2] = b.x; f[3] = b.y;
}
template <typename T> __device__ __forceinline__ void st4(T* p, const float* f);
template <> __device__ __forceinline__ void st4<float>(float* p, const float* f) {
  *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]);
}
template <> __device__ __forceinline__ void st4<bf16>(bf16* p, const float* f) {
  __nv_bfloat162 a = __floats2bfloat162_rn(f[0], f[1]), b = __floats2bfloat162_rn(f[2], f[3]);
  uint2 v;
  v.x = *reinterpret_cast<uint32_t*>(&a);
  v.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = v;
}
// sum += p[s * stride] over all s, in index order: up to AHEAD slots are requested before the first is added.  (Left to the
// compiler's unrolling by four, slots beyond a multiple of four were a round trip to L2 each.  64 rows of a 4096-wide model, behind the kernel in front:
// norm of ten slots 6.1 -> 4.7 us, of five 4.0.  A spilled register costs more than a round trip gains.)  p is the same for all threads of a block, so that only `col` (in floats) takes registers.
template <int AHEAD, int COLS>
__device__ __forceinline__ void add_slots(float4 (&sum)[COLS], const float* p, const uint32_t (&col)[COLS], int nsplit, size_t stride) {
#pragma unroll 1
  for (int s0 = 0; s0 < nsplit; s0 += AHEAD) {
    float4 t[AHEAD][COLS];
#pragma unroll
    for (int u = 0; u < AHEAD; ++u, p += stride)
      if (s0 + u < nsplit)
#pragma unroll
        for (int c = 0; c < COLS; ++c) t[u][c] = *reinterpret_cast<const float4*>(p + col[c]);
#pragma unroll
    for (int u = 0; u < AHEAD; ++u)
      if (s0 + u < nsplit)
#pragma unroll
        for (int c = 0; c < COLS; ++c) { sum[c].x += t[u][c].x; sum[c].y += t[u][c].y; sum[c].z += t[u][c].z; sum[c].w += t[u][c].w; }
  }
}
// One row per CTA, four consecutive columns per thread:
//   x <- (embedding row | x | x + sum of GEMM partial slots), kept in fp32 (the residual stream is never rounded);
//   out <- RMSNorm(x) * gain, in the model's storage type.
// Fusing the residual add (and the first layer's embedding gather) with the norm that always follows
// it halves the element-wise launches.  Of up to 8192 columns, all of up to eight slots of a thread's columns are on their way at once
// (four or five after a product of 64 rows), above that two.  The sums of the warps are read back four at a time.
constexpr int NORM_THREADS = 1024;
constexpr int NORM_MAX_ITER = 4;          // d_model up to 16384
template <typename T, int ITER, int AHEAD, int THREADS = NORM_THREADS>
__global__ void __launch_bounds__(THREADS, NORM_THREADS / THREADS) fused_norm_kernel(float* __restrict__ x, const float* part, int nsplit,
                                                                   size_t split_stride, const T* __restrict__ embed,
                                                                   const int32_t* tok, int tok_stride, int tok_off,
                                                                   const int32_t* n_active, int n, int V,
                                                                   const T* __restrict__ gain, T* __restrict__ out, int d, float eps,
                                                                   const int32_t* row_off, int B) {
  __shared__ __align__(16) float red[32];
  const int row = blockIdx.x;
  float* xr = x + (size_t)row * d;
  // The residual stream was last written by the previous norm (at least two kernels ago) and the gains
  // never change: both are fetched before waiting for the kernel in front (a GEMM, or whatever produced
  // the token ids), so that after the wait only that kernel's output remains to be read.
  float keep[ITER][4], gv[ITER][4];
#pragma unroll
  for (int it = 0; it < ITER; ++it) {
    const int j = (it * THREADS + threadIdx.x) * 4;
    if (j < d) {
      if (!embed) ld4(xr + j, keep[it]);
      if (out) ld4(gain + j, gv[it]);
    }
  }
  griddep_wait();
  griddep_launch();
  const T* src = nullptr;
  if (embed) {
    int b, v, t = 0;
    locate_row(row, row_off, B, n, b, v);
    if (v < n_active[b]) t = tok[(size_t)b * tok_stride + tok_off + v];
    if (t < 0 || t >= V) t = 0;
    src = embed + (size_t)t * d;
  }
  float ss = 0.f;
#pragma unroll
  for (int it = 0; it < ITER; ++it) {
    const int j = (it * THREADS + threadIdx.x) * 4;
    if (j < d) {
      float v[4];
      if (src) ld4(src + j, v);
      else {
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = keep[it][e];
      }
      if (nsplit > 0) {
        float4 sum[1] = {make_float4(0.f, 0.f, 0.f, 0.f)};
        add_slots<AHEAD>(sum, part + (size_t)row * d, {(uint32_t)j}, nsplit, split_stride);
        const float4 a = sum[0];
        v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w;
      }
      if (embed || nsplit > 0) st4(xr + j, v);
#pragma unroll
      for (int e = 0; e < 4; ++e) { keep[it][e] = v[e]; ss += v[e] * v[e]; }
    }
  }
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  ss = 0.f;
#pragma unroll
  for (int w = 0; w < THREADS / 32; w += 4) {
    const float4 r4 = *reinterpret_cast<const float4*>(red + w);
    ss += r4.x; ss += r4.y; ss += r4.z; ss += r4.w;
  }
  if (!out) return;
  const float r = 1.0f / sqrtf(ss / (float)d + eps);
  T* o = out + (size_t)row * d;
#pragma unroll
  for (int it = 0; it < ITER; ++it) {
    const int j = (it * THREADS + threadIdx.x) * 4;
    if (j < d) {
      float ov[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) ov[e] = keep[it][e] * r * gv[it][e];
      st4(o + j, ov);
    }
  }
}

// The same without slots (the GEMMs add to the residual stream themselves, so it is read after the wait).  Many rows are memory-bound: eight CTAs of 256 threads to an SM.  (One 1024-thread CTA per SM and row: 33 us for 2048 rows of 4096 where the bytes take 8.)
constexpr int ROWS_THREADS = 256;
template <typename T, int ITER>
__global__ void __launch_bounds__(ROWS_THREADS) row_norm_kernel(float* x, const T* __restrict__ embed, const int32_t* tok,
                                                                int tok_stride, int tok_off, const int32_t* n_active, int n, int V,
                                                                const T* __restrict__ gain, T* __restrict__ out, int d, float eps,
                                                                const int32_t* row_off, int B) {
  __shared__ float red[32];
  const int row = blockIdx.x;
  griddep_wait();
  griddep_launch();
  float* xr = x + (size_t)row * d;
  const T* src = nullptr;
  if (embed) {
    int b, v, t = 0;
    locate_row(row, row_off, B, n, b, v);
    if (v < n_active[b]) t = tok[(size_t)b * tok_stride + tok_off + v];
    if (t < 0 || t >= V) t = 0;
    src = embed + (size_t)t * d;
  }
  float v[ITER][4];
#pragma unroll
  for (int it = 0; it < ITER; ++it) {
    const int j = (it * ROWS_THREADS + threadIdx.x) * 4;
    v[it][0] = v[it][1] = v[it][2] = v[it][3] = 0.f;
    if (j < d) {
      if (src) ld4(src + j, v[it]);
      else ld4(xr + j, v[it]);
    }
  }
  float ss = 0.f;
#pragma unroll
  for (int it = 0; it < ITER; ++it) {
    const int j = (it * ROWS_THREADS + threadIdx.x) * 4;
    if (src && j < d) st4(xr + j, v[it]);
#pragma unroll
    for (int e = 0; e < 4; ++e) ss += v[it][e] * v[it][e];
  }
  ss = block_sum(ss, red);
  const float r = 1.0f / sqrtf(ss / (float)d + eps);
  T* o = out + (size_t)row * d;
#pragma unroll
  for (int it = 0; it < ITER; ++it) {
    const int j = (it * ROWS_THREADS + threadIdx.x) * 4;
    if (j < d) {
      float g[4], ov[4];
      ld4(gain + j, g);
#pragma unroll
      for (int e = 0; e < 4; ++e) ov[e] = v[it][e] * r * g[e];
      st4(o + j, ov);
    }
  }
}

// q,k rotated at position len + depth; k,v stored at slot len + node of the paged pools; q kept dense.
// One CTA per (row, head), one thread per rotation pair.
template <typename T>
__global__ void rope_append_kernel(const float* part, int nsplit, size_t split_stride,
                                   const int32_t* __restrict__ len, const int32_t* __restrict__ n_active,
                                   const int32_t* __restrict__ depth, const int32_t* __restrict__ page_table,
                                   int max_pages, const float2* __restrict__ rope, int max_pos, int n, int H, int Dh,
                                   T* __restrict__ q, T* __restrict__ kpool, T* __restrict__ vpool,
                                   const int32_t* __restrict__ row_off, int B) {
  // Lengths, live node counts, the tree, the page table and the rotation table are at least two kernels
  // old: the chain of dependent index loads runs before the wait for the QKV GEMM in front.
  const int row = blockIdx.x, h = blockIdx.y;
  int b, v;
  locate_row(row, row_off, B, n, b, v);          // (the row offsets come from the host, before the step's first kernel)
  const int HD = H * Dh, half = Dh >> 1;
  const bool active = v < n_active[b];
  const int L = len[b];
  const int pos = L + depth[v], slot = L + v;
  const bool ok = active && pos < max_pos && slot < max_pos;
  const int page = ok ? page_table[(size_t)b * max_pages + slot / CERB_PAGE] : 0;
  const float2 cs0 = (ok && (int)threadIdx.x < half) ? rope[(size_t)pos * half + threadIdx.x] : make_float2(1.f, 0.f);
  griddep_wait();
  griddep_launch();
  if (!ok) return;
  const size_t kv = (((size_t)page * H + h) * CERB_PAGE + (size_t)(slot % CERB_PAGE)) * Dh;
  const float* pr = part + (size_t)row * 3 * HD + h * Dh;
  for (int i = threadIdx.x; i < half; i += blockDim.x) {
    float2 cs = i == (int)threadIdx.x ? cs0 : rope[(size_t)pos * half + i];
    float sum[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};          // q, k, v: the pair's two columns each
    constexpr int AHEAD = 4;                                 // (the slots of a 12288-column product of 64 rows: on their way at once)
    const float* p = pr + i;
#pragma unroll 1
    for (int s0 = 0; s0 < nsplit; s0 += AHEAD) {
      float t[AHEAD][6];
#pragma unroll
      for (int u = 0; u < AHEAD; ++u, p += split_stride)
        if (s0 + u < nsplit) {
          t[u][0] = p[0]; t[u][1] = p[half]; t[u][2] = p[HD]; t[u][3] = p[HD + half]; t[u][4] = p[2 * HD]; t[u][5] = p[2 * HD + half];
        }
#pragma unroll
      for (int u = 0; u < AHEAD; ++u)
        if (s0 + u < nsplit)
#pragma unroll
          for (int c = 0; c < 6; ++c) sum[c] += t[u][c];
    }
    const float q1 = sum[0], q2 = sum[1], k1 = sum[2], k2 = sum[3], v1 = sum[4], v2 = sum[5];
    T* qo = q + (size_t)row * HD + h * Dh + i;
    stf(qo, q1 * cs.x - q2 * cs.y);
    stf(qo + half, q2 * cs.x + q1 * cs.y);
    stf(kpool + kv + i, k1 * cs.x - k2 * cs.y);
    stf(kpool + kv + i + half, k2 * cs.x + k1 * cs.y);
    stf(vpool + kv + i, v1);
    stf(vpool + kv + i + half, v2);
  }
}

template <typename T, int AHEAD>
__global__ void swiglu_kernel(const float* part, int nsplit, size_t split_stride, T* __restrict__ act, int F) {
  const size_t row = blockIdx.x;
  const int j = (blockIdx.y * blockDim.x + threadIdx.x) * 4;
  griddep_wait();
  griddep_launch();
  if (j >= F) return;
  float4 gu[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
  add_slots<AHEAD>(gu, part + row * 2 * F, {(uint32_t)j, (uint32_t)(F + j)}, nsplit, split_stride);
  const float4 g = gu[0], u = gu[1];
  T* o = act + row * F + j;
  stf(o, g.x / (1.0f + expf(-g.x)) * u.x);
  stf(o + 1, g.y / (1.0f + expf(-g.y)) * u.y);
  stf(o + 2, g.z / (1.0f + expf(-g.z)) * u.z);
  stf(o + 3, g.w / (1.0f + expf(-g.w)) * u.w);
}

// Row argmax over logits given as split-K partial sums; ties go to the lower index.  When
// `summed` is not null the summed logits are also written there ([rows][V]).
// A thread has U groups of four columns in S slots each on their way at once.
template <int U, int S>
__global__ void __launch_bounds__(1024) argmax_rows_kernel(const float* part, int nsplit, size_t split_stride, int V,
                                   int32_t* __restrict__ out, float* __restrict__ summed) {
  __shared__ float sv[32];
  __shared__ int si[32];
  griddep_wait();
  griddep_launch();
  const float* r = part + (size_t)blockIdx.x * V;
  float best = -INFINITY;
  int bi = 0x7fffffff;
  if ((V & 3) == 0 && (split_stride & 3) == 0) {
    const int V4 = V >> 2;
    for (int base = threadIdx.x; base < V4; base += U * blockDim.x) {
      float4 a[U];
#pragma unroll
      for (int u = 0; u < U; ++u) a[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      // (columns past the row's end read its last ones again and are not looked at)
      uint32_t col[U];
#pragma unroll
      for (int u = 0; u < U; ++u) col[u] = 4 * min(base + u * (int)blockDim.x, V4 - 1);
      add_slots<S>(a, r, col, nsplit, split_stride);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j4 = base + u * blockDim.x;
        if (j4 >= V4) break;
        if (summed) *reinterpret_cast<float4*>(summed + (size_t)blockIdx.x * V + 4 * j4) = a[u];
        const int j = 4 * j4;                     // ascending ids: a later equal value never replaces an earlier one
        if (a[u].x > best) { best = a[u].x; bi = j; }
        if (a[u].y > best) { best = a[u].y; bi = j + 1; }
        if (a[u].z > best) { best = a[u].z; bi = j + 2; }
        if (a[u].w > best) { best = a[u].w; bi = j + 3; }
      }
    }
  } else {
    for (int j = threadIdx.x; j < V; j += blockDim.x) {
      float v = 0.f;
      for (int s = 0; s < nsplit; ++s) v += r[s * split_stride + j];
      if (summed) summed[(size_t)blockIdx.x * V + j] = v;
      if (v > best || (v == best && j < bi)) { best = v; bi = j; }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    float ov = __shfl_xor_sync(0xffffffffu, best, o);
    int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
  }
  int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (l == 0) { sv[w] = best; si[w] = bi; }
  __syncthreads();
  if (w == 0) {
    best = l < nw ? sv[l] : -INFINITY;
    bi = l < nw ? si[l] : 0x7fffffff;
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    if (l == 0) out[blockIdx.x] = (bi == 0x7fffffff) ? 0 : bi;
  }
}

// mode 0: n_active[b] = a.  mode 1 (prefill chunk): n_active[b] = clamp(lens_in[b] - a, 0, b_), and row_off[b] = the first
// of the rows that sequence b owns when only live tokens have rows.
__global__ void set_nactive_kernel(int32_t* n_active, const int32_t* lens_in, int32_t* row_off, int B, int mode, int a, int b_) {
  griddep_wait();
  griddep_launch();
  const int b = threadIdx.x;
  int r = 0;
  if (b < B) {
    r = a;
    if (mode == 1) {
      r = lens_in[b] - a;
      r = r < 0 ? 0 : (r > b_ ? b_ : r);
    }
    n_active[b] = r;
  }
  if (mode == 1) {
    int sum = r;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, sum, o);
      if (b >= o) sum += t;
    }
    if (b <= B) row_off[b] = sum - r;
  }
}

// After a chain-shaped prefill chunk: everything is accepted in place.
template <typename T>
__global__ void prefill_commit_kernel(const int32_t* n_active, int32_t* len, const T* hidden, T* __restrict__ h_last, const int32_t* row_off, int d) {
  griddep_wait();
  griddep_launch();
  int b = blockIdx.x, na = n_active[b];
  if (na <= 0) return;
  const T* src = hidden + ((size_t)row_off[b] + na - 1) * d;
  for (int j = threadIdx.x; j < d; j += blockDim.x) h_last[(size_t)b * d + j] = src[j];
  __syncthreads();
  if (threadIdx.x == 0) len[b] += na;
}

int launch_rope_table(cerb_ctx* c, cudaStream_t st) {
  int half = c->cfg.head_dim / 2, total = c->max_pos * half;
  rope_table_kernel<<<(total + 255) / 256, 256, 0, st>>>(c->d_rope, c->max_pos, half, (double)c->cfg.rope_base);
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

// x <- embedding rows (tok != null) | x + partials (nsplit > 0) | x;  out <- RMSNorm(x) * gain (out may be null).
// complete: the forward's GEMMs add to the residual stream themselves.
int launch_fused_norm(cerb_ctx* c, const float* part, int nsplit, size_t split_stride, const int32_t* tok, int tok_stride,
                      int tok_off, int n, const void* gain, void* out, int rows, cudaStream_t st, const int32_t* row_off,
                      bool complete) {
  const cerb_config& g = c->cfg;
  const int d = g.d_model;
  if (d % 4 || d > NORM_THREADS * NORM_MAX_ITER * 4) return CERB_E_SHAPE;
  if (complete && nsplit == 0 && out) {
    auto rows_of = [&](auto type, auto iter) {
      typedef decltype(type) T;
      launch_pdl(row_norm_kernel<T, decltype(iter)::value>, dim3(rows), dim3(ROWS_THREADS), 0, st, (float*)c->d_x,
                 tok ? (const T*)c->embed : (const T*)nullptr, tok, tok_stride, tok_off, (const int32_t*)c->d_nactive, n, g.vocab,
                 (const T*)gain, (T*)out, d, g.rms_eps, row_off, c->B);
    };
    auto wide = [&](auto iter) { c->bf16 ? rows_of(bf16(), iter) : rows_of(float(), iter); };
    if (d <= 4096) wide(std::integral_constant<int, 4>());
    else if (d <= 8192) wide(std::integral_constant<int, 8>());
    else wide(std::integral_constant<int, 16>());
  } else {
    auto go = [&](auto kern, auto type, int threads = NORM_THREADS) {
      typedef decltype(type) T;
      launch_pdl(kern, dim3(rows), dim3(threads), 0, st, (float*)c->d_x, part, nsplit, split_stride,
                 tok ? (const T*)c->embed : (const T*)nullptr, tok, tok_stride, tok_off, (const int32_t*)c->d_nactive, n, g.vocab,
                 (const T*)gain, (T*)out, d, g.rms_eps, row_off, c->B);
    };
    // Products of gemm_rows.cu leave at most eight slots: of up to 8192 columns they are one trip to L2; wider rows take two at a time.  (Matrices that it does not take,
    // of fewer than 16 rows per SM and part of k, leave up to 16: two trips and more.)  More rows than SMs, with slots: two blocks of half the
    // threads to an SM (256 rows of 4096 / 5120 columns 6.7 / 7.6 -> 5.0 / 5.0 us; without slots 2048-row forwards of 4096 columns took 26.14 ms so and 26.00 with one block).
    const bool one = d <= NORM_THREADS * 4;
    if (c->bf16 && nsplit > 0 && rows > c->sm_count && one) go(fused_norm_kernel<bf16, 2, 4, NORM_THREADS / 2>, bf16(), NORM_THREADS / 2);
    else if (c->bf16 && nsplit > 0 && rows > c->sm_count && d <= NORM_THREADS * 6) go(fused_norm_kernel<bf16, 3, 4, NORM_THREADS / 2>, bf16(), NORM_THREADS / 2);
    else if (c->bf16 && one) go(fused_norm_kernel<bf16, 1, 8>, bf16());
    else if (c->bf16 && d <= NORM_THREADS * 8) go(fused_norm_kernel<bf16, 2, 8>, bf16());
    else if (c->bf16) go(fused_norm_kernel<bf16, NORM_MAX_ITER, 2>, bf16());
    else if (one) go(fused_norm_kernel<float, 1, 8>, float());
    else go(fused_norm_kernel<float, NORM_MAX_ITER, 2>, float());
  }
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

int launch_rope_append(cerb_ctx* c, int layer, const TreeDev& t, const float* part, int nsplit, size_t split_stride,
                       int B, int n, int rows, cudaStream_t st, const int32_t* row_off) {
  const cerb_config& g = c->cfg;
  char* kp = c->k_pool + (size_t)layer * c->pool_layer_bytes;
  char* vp = c->v_pool + (size_t)layer * c->pool_layer_bytes;
  if (c->bf16)
    launch_pdl(rope_append_kernel<bf16>, dim3(rows, g.n_heads), dim3(64), 0, st, part, nsplit, split_stride,
               (const int32_t*)c->d_len, (const int32_t*)c->d_nactive, (const int32_t*)t.depth, c->page_table, g.max_pages,
               (const float2*)c->d_rope, c->max_pos, n, g.n_heads, g.head_dim, (bf16*)c->d_q, (bf16*)kp, (bf16*)vp, row_off, B);
  else
    launch_pdl(rope_append_kernel<float>, dim3(rows, g.n_heads), dim3(64), 0, st, part, nsplit, split_stride,
               (const int32_t*)c->d_len, (const int32_t*)c->d_nactive, (const int32_t*)t.depth, c->page_table, g.max_pages,
               (const float2*)c->d_rope, c->max_pos, n, g.n_heads, g.head_dim, (float*)c->d_q, (float*)kp, (float*)vp, row_off, B);
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

int launch_swiglu(cerb_ctx* c, const float* part, int nsplit, size_t split_stride, void* act, int rows, cudaStream_t st) {
  const int F = c->cfg.mlp_dim;
  const dim3 grid(rows, (F / 4 + 255) / 256);
  // Three slots at once (4096 columns and wider); four take 16 registers more, which three slots would only pay for (six layers of 4096 x
  // 11008, 64 rows: 682 and 689 us) and four need (2048 x 5632, 64 rows: 4.2 -> 3.2 us; 3.8 unrolled by four).
  if (!c->bf16) launch_pdl(swiglu_kernel<float, 3>, grid, dim3(256), 0, st, part, nsplit, split_stride, (float*)act, F);
  else if (nsplit <= 3) launch_pdl(swiglu_kernel<bf16, 3>, grid, dim3(256), 0, st, part, nsplit, split_stride, (bf16*)act, F);
  else launch_pdl(swiglu_kernel<bf16, 4>, grid, dim3(256), 0, st, part, nsplit, split_stride, (bf16*)act, F);
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

int launch_argmax_rows(cerb_ctx* c, const float* part, int nsplit, size_t split_stride, int rows, int V, int32_t* out,
                       float* summed, cudaStream_t st) {
  // One slot: a row of 32000 columns is on its way at once where SMs are left over; else as many threads as let all rows in at once, or
  // four rows to an SM, the loads of one beside the reduction of another (2048 rows: 97 -> 67 us; 256 rows 9.0 -> 6.3; one row 4.4 -> 3.5, 64 rows of three
  // slots 8.2 -> 7.4).
  auto go = [&](auto kern, int threads) { launch_pdl(kern, dim3(rows), dim3(threads), 0, st, part, nsplit, split_stride, V, out, summed); };
  if (nsplit == 1) go(argmax_rows_kernel<8, 1>, rows <= c->sm_count ? 1024 : rows <= 2 * c->sm_count ? 512 : 256);
  else if (nsplit == 2) go(argmax_rows_kernel<4, 2>, 1024);
  else go(argmax_rows_kernel<2, 3>, 1024);
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

int launch_set_nactive(cerb_ctx* c, int mode, int a, int b, cudaStream_t st) {
  set_nactive_kernel<<<1, 32, 0, st>>>(c->d_nactive, c->d_lens_in, c->d_rowoff, c->B, mode, a, b);
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

int launch_prefill_commit(cerb_ctx* c, cudaStream_t st) {
  int d = c->cfg.d_model;
  if (c->bf16)
    prefill_commit_kernel<bf16><<<c->B, 256, 0, st>>>(c->d_nactive, c->d_len, (const bf16*)c->d_hidden,
                                                      (bf16*)c->d_hlast, (const int32_t*)c->d_rowoff, d);
  else
    prefill_commit_kernel<float><<<c->B, 256, 0, st>>>(c->d_nactive, c->d_len, (const float*)c->d_hidden,
                                                       (float*)c->d_hlast, (const int32_t*)c->d_rowoff, d);
  CERB_LAUNCH_CHECK(c);
  return CERB_OK;
}

}  // namespace cerb
