// Memory-bound and control kernels of the Amphista step: embedding, fused residual + RMSNorm,
// rotary embedding + KV write, split-KV tree attention with a bitmask, SwiGLU, the draft
// module's head kernels (Eq. 2-6), tree construction, greedy acceptance and KV compaction.
#include <math.h>

#include "amph_internal.cuh"

namespace amph {

typedef __nv_bfloat16 bf16;

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(bf16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T from_f(float v);
template <> __device__ __forceinline__ float from_f<float>(float v) { return v; }
template <> __device__ __forceinline__ bf16 from_f<bf16>(float v) { return __float2bfloat16_rn(v); }

#define AMPH_DISPATCH(dtype, ...)                                    \
  do {                                                               \
    if ((dtype) == AMPH_DTYPE_F32) { typedef float T; __VA_ARGS__; } \
    else { typedef bf16 T; __VA_ARGS__; }                            \
  } while (0)

__device__ __forceinline__ float sum_partials(const PartialView& P, int row, int col) {
  const float* p = P.p + (size_t)row * P.ld + col;
  float acc = p[0];
  for (int s = 1; s < P.splits; ++s) acc += p[(size_t)s * P.split_stride];   // fixed order: deterministic
  return acc;
}

// The partial sums sit in L2, one round trip each: the loads of a batch of N splits are issued together,
// then added in split order.
template <int N>
__device__ __forceinline__ void add_splits(const float* p, size_t stride, int s0, int splits, float4& acc) {
  float4 v[N];
#pragma unroll
  for (int s = 0; s < N; ++s)
    if (s0 + s < splits) v[s] = *reinterpret_cast<const float4*>(p + (size_t)(s0 + s) * stride);
#pragma unroll
  for (int s = 0; s < N; ++s)
    if (s0 + s < splits) { acc.x += v[s].x; acc.y += v[s].y; acc.z += v[s].z; acc.w += v[s].w; }
}

// Same sum for kernels with registers to spare and many splits to read (the residual kernels).
__device__ __forceinline__ float4 sum_partials4_wide(const PartialView& P, int row, int col) {
  const float* p = P.p + (size_t)row * P.ld + col;
  float4 acc = *reinterpret_cast<const float4*>(p);
  const int n = P.splits;
  if (n == 1) return acc;
  for (int s0 = 1; s0 < n; s0 += 8) add_splits<8>(p, P.split_stride, s0, n, acc);
  return acc;
}

__device__ __forceinline__ void store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(bf16* p, float4 v) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  uint2 u;
  u.x = *reinterpret_cast<unsigned*>(&a);
  u.y = *reinterpret_cast<unsigned*>(&b);
  *reinterpret_cast<uint2*>(p) = u;
}
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const bf16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16),
                     __uint_as_float(u.y & 0xffff0000u));
}

__device__ __forceinline__ float block_sum(float v, float* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  float t = 0.f;
  for (int i = 0; i < nw; ++i) t += red[i];
  return t;
}

// --------------------------------------------------------------------------------------------
// residual update + RMSNorm (one block per row)
// --------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(1024)
resid_norm_kernel(float* __restrict__ x, PartialView P, int col_off, int mode, const T* __restrict__ gain,
                  T* __restrict__ xn, float* __restrict__ hid, float eps, int d) {
  pdl_wait();
  pdl_launch_dependents();
  extern __shared__ __align__(16) float rowbuf[];
  __shared__ float red[32];
  const int r = blockIdx.x;
  float* xr = x + (size_t)r * d;
  float ss = 0.f;
  for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4) {
    float4 v;
    if (mode == 0) {
      v = load4(xr + c);
    } else {
      v = sum_partials4(P, r, col_off + c);
      if (mode == 1) { const float4 o = load4(xr + c); v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w; }
      store4(xr + c, v);
    }
    store4(rowbuf + c, v);
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
  if (xn == nullptr && hid == nullptr) return;
  if (gain == nullptr) {                       // plain cast of the updated row (each thread re-reads its own chunk)
    for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4) {
      const float4 v = load4(rowbuf + c);
      if (xn) store4(xn + (size_t)r * d + c, v);
      if (hid) store4(hid + (size_t)r * d + c, v);
    }
    return;
  }
  const float tot = block_sum(ss, red);
  const float inv = 1.0f / sqrtf(tot / (float)d + eps);
  for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4) {
    const float4 v = load4(rowbuf + c), g = load4(gain + c);
    const float4 n = make_float4(g.x * (v.x * inv), g.y * (v.y * inv), g.z * (v.z * inv), g.w * (v.w * inv));
    if (xn) store4(xn + (size_t)r * d + c, n);
    if (hid) store4(hid + (size_t)r * d + c, n);
  }
}

void launch_resid_norm(float* x, PartialView P, int col_off, int mode, const void* gain, int dtype,
                       void* xn, float* hid, float eps, int rows, int d, cudaStream_t st) {
  int threads = (d / 4 + 31) / 32 * 32;
  if (threads > 1024) threads = 1024;
  AMPH_DISPATCH(dtype, launch_pdl(resid_norm_kernel<T>, dim3(rows), dim3(threads), d * sizeof(float), st, 
                           x, P, col_off, mode, (const T*)gain, (T*)xn, hid, eps, d));
}

// Residual update without the row-wide reduction: grid (row, 512-column chunk).  The division by the row's
// RMS is left to the kernel that consumes the next projection (RowScale), so every block is independent.
template <typename T>
__global__ void __launch_bounds__(128)
resid_scale_kernel(float* __restrict__ x, PartialView P, int col_off, int mode, const T* __restrict__ gain,
                   T* __restrict__ xn, float* __restrict__ ss_part, int d, int early) {
  if (early) pdl_launch_dependents();
  pdl_wait();
  if (!early) pdl_launch_dependents();
  __shared__ float red[32];
  const int r = blockIdx.x;
  const int c = blockIdx.y * kScaleChunkCols + threadIdx.x * 4;
  float ss = 0.f;
  if (c < d) {
    float* xr = x + (size_t)r * d + c;
    float4 v = sum_partials4_wide(P, r, col_off + c);
    if (mode == 1) { const float4 o = load4(xr); v.x += o.x; v.y += o.y; v.z += o.z; v.w += o.w; }
    store4(xr, v);
    if (gain != nullptr) {
      const float4 g = load4(gain + c);
      store4(xn + (size_t)r * d + c, make_float4(g.x * v.x, g.y * v.y, g.z * v.z, g.w * v.w));
      ss = v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    }
  }
  if (gain == nullptr) return;
  const float tot = block_sum(ss, red);
  if (threadIdx.x == 0) ss_part[r * gridDim.y + blockIdx.y] = tot;
}

void launch_resid_scale(float* x, PartialView P, int col_off, int mode, const void* gain, int dtype, void* xn,
                        float* ss_part, int rows, int d, cudaStream_t st, int early) {
  const int chunks = (d + kScaleChunkCols - 1) / kScaleChunkCols;
  AMPH_DISPATCH(dtype, launch_pdl(resid_scale_kernel<T>, dim3(rows, chunks), dim3(128), 0, st, x, P, col_off, mode,
                                  (const T*)gain, (T*)xn, ss_part, d, early));
}

// --------------------------------------------------------------------------------------------
// start of a pass: row tables, rotary tables, and the rows themselves
// --------------------------------------------------------------------------------------------
__device__ __forceinline__ void chain_mask(int r, u64* m) {       // bits 0..r
  m[0] = r >= 63 ? ~0ull : ((1ull << (r + 1)) - 1ull);
  m[1] = r < 64 ? 0ull : (r >= 127 ? ~0ull : ((1ull << (r - 63)) - 1ull));
}

// Row `rl` of group g: its rotary table row, and (row 0 of a chain) the group's whole row table.  A chain is a run of tokens
// at consecutive positions, each seeing the ones before it: prompt chunks, or the rows an adaptation layer has pending.
__device__ __forceinline__ void setup_row(const PassRows& p, int g, int rl) {
  RowMeta* meta = reinterpret_cast<RowMeta*>(p.meta + p.meta_stride * g);
  int pos;
  if (p.source == PassRows::kTree) {                             // the table was written with the tree
    pos = meta->pos[rl];
  } else {
    int base = p.base[g], n = p.n[g];
    if (p.source == PassRows::kPending) {
      const DevState* s = reinterpret_cast<const DevState*>(p.state + p.state_stride * g);
      n = s->n_pending;
      n = n < 0 ? 0 : (n > kPendMax ? kPendMax : n);
      base = s->C - n;
    }
    pos = base + rl;
    if (rl == 0) {
      if (threadIdx.x == 0) { meta->base = base; meta->n_rows = n; }
      for (int r = threadIdx.x; r < kMaxRows; r += blockDim.x) {
        meta->pos[r] = base + r;
        meta->slot[r] = base + r;
        chain_mask(r, meta->mask[r]);
      }
    }
  }
  // table[r][i] = (cos, sin)(pos * theta^(-2i/dh)), in double: positions of thousands leave no room for a float angle
  float2* table = reinterpret_cast<float2*>(p.rope + p.rope_stride * g) + (size_t)rl * p.half;
  for (int i = threadIdx.x; i < p.half; i += blockDim.x) {
    double sn, cs;
    sincos((double)pos * p.inv_freq[i], &sn, &cs);
    table[i] = make_float2((float)cs, (float)sn);
  }
}

// Start of a target pass, one block per row: row set-up, x = the token's embedding, xn = its RMSNorm with the first layer's
// gain, in one launch for all groups.  Latency: a launch of its own for each costs 1.2-1.8 us of the chain, per group for the
// tables (six launches fewer per step: 275 -> 269 us on a three-layer model of width 512).  A chain's row table is read by the attention kernel before its dependency wait, and the projection between lets
// that kernel start at once: such a pass triggers its successor only by ending.
template <typename T>
__global__ void __launch_bounds__(1024)
target_rows_kernel(const PassRows p, const T* __restrict__ emb, const int* __restrict__ toks, int vocab, int d,
                   const T* __restrict__ gain, float eps, float* __restrict__ x, T* __restrict__ xn) {
  pdl_wait();
  if (p.source == PassRows::kTree) pdl_launch_dependents();
  extern __shared__ __align__(16) float rowbuf[];
  __shared__ float red[32];
  const int r = blockIdx.x, g = r / p.rpg;
  if (r == 0 && p.clear != nullptr)
    for (int i = threadIdx.x; i < p.n_clear; i += blockDim.x) p.clear[i] = 0;
  int t = toks[r];
  t = t < 0 ? 0 : (t >= vocab ? vocab - 1 : t);
  const T* e = emb + (size_t)t * d;
  float ss = 0.f;
  for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4) {
    const float4 v = load4(e + c);
    store4(x + (size_t)r * d + c, v);
    store4(rowbuf + c, v);
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
  setup_row(p, g, r - g * p.rpg);
  const float inv = 1.0f / sqrtf(block_sum(ss, red) / (float)d + eps);
  for (int c = threadIdx.x * 4; c < d; c += blockDim.x * 4) {
    const float4 v = load4(rowbuf + c), w = load4(gain + c);
    store4(xn + (size_t)r * d + c, make_float4(w.x * (v.x * inv), w.y * (v.y * inv), w.z * (v.z * inv), w.w * (v.w * inv)));
  }
}

void launch_target_rows(const PassRows& p, int G, const void* tok_emb, int dtype, const int* toks, int vocab, int d, const void* gain,
                        float eps, float* x, void* xn, cudaStream_t st) {
  int threads = (d / 4 + 31) / 32 * 32;
  if (threads > 1024) threads = 1024;
  AMPH_DISPATCH(dtype, launch_pdl(target_rows_kernel<T>, dim3(G * p.rpg), dim3(threads), d * sizeof(float), st, p, (const T*)tok_emb, toks,
                                  vocab, d, (const T*)gain, eps, x, (T*)xn));
}

// Start of an adaptation stage (Eq. 1), all groups: cat[r] = [feature ; embedding of the next token], and for the first stage
// (setup != 0) the pass's row set-up.  emb == NULL: the ablation without the sampled token; the row is the feature alone.
template <typename T>
__global__ void __launch_bounds__(256)
sal_rows_kernel(const PassRows p, int setup, const float* __restrict__ feat, const T* __restrict__ emb, const char* next_tok,
                size_t next_stride, int vocab, T* __restrict__ cat, int d) {
  pdl_wait();
  pdl_launch_dependents();
  const int r = blockIdx.x, g = r / p.rpg, rl = r - g * p.rpg;
  const size_t pitch = emb ? 2 * (size_t)d : (size_t)d;
  int t = reinterpret_cast<const int*>(next_tok + next_stride * g)[rl];
  t = t < 0 ? 0 : (t >= vocab ? vocab - 1 : t);
  for (int c = (blockIdx.y * blockDim.x + threadIdx.x) * 4; c < d; c += gridDim.y * blockDim.x * 4) {
    store4(cat + (size_t)r * pitch + c, load4(feat + (size_t)r * d + c));
    if (emb) store4(cat + (size_t)r * pitch + d + c, load4(emb + (size_t)t * d + c));
  }
  if (setup && blockIdx.y == 0) setup_row(p, g, rl);
}

void launch_sal_rows(const PassRows& p, int G, int setup, const float* feat, const void* tok_emb, const void* next_tok, size_t next_stride,
                     int vocab, void* cat, int dtype, int d, cudaStream_t st) {
  const int gy = (d / 4 + 255) / 256;
  AMPH_DISPATCH(dtype, launch_pdl(sal_rows_kernel<T>, dim3(G * p.rpg, gy), dim3(256), 0, st, p, setup, feat, (const T*)tok_emb,
                                  (const char*)next_tok, next_stride, vocab, (T*)cat, d));
}

// --------------------------------------------------------------------------------------------
// q / k rotation, KV-cache write (one block per row)
// --------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256)
qkv_rope_kernel(PartialView P, const RowMeta* __restrict__ meta, const float2* __restrict__ rope, T* __restrict__ q,
                T* __restrict__ kc, T* __restrict__ vc, int n_heads, int dh, int max_ctx, RowScale rs) {
  pdl_wait();
  pdl_launch_dependents();
  const int r = blockIdx.x;
  const int half = dh >> 1, d = n_heads * dh, quads = half >> 2;
  const bool live = r < meta->n_rows;
  const int slot = meta->slot[r];
  const bool store = live && slot >= 0 && slot < max_ctx;
  const float sc = row_scale(rs, r);
  // one item = four rotation pairs (i..i+3, i+half..) of one head; grid.y strides over the items of the row
  for (int idx = blockIdx.y * blockDim.x + threadIdx.x; idx < n_heads * quads; idx += gridDim.y * blockDim.x) {
    const int h = idx / quads, i = (idx - h * quads) * 4;
    const float4 cs0 = *reinterpret_cast<const float4*>(rope + r * half + i);       // (c0,s0,c1,s1)
    const float4 cs1 = *reinterpret_cast<const float4*>(rope + r * half + i + 2);   // (c2,s2,c3,s3)
    const int c0 = h * dh + i, c1 = c0 + half;
    {
      float4 a = sum_partials4(P, r, c0), b = sum_partials4(P, r, c1);
      a.x *= sc; a.y *= sc; a.z *= sc; a.w *= sc; b.x *= sc; b.y *= sc; b.z *= sc; b.w *= sc;
      store4(q + (size_t)r * d + c0, make_float4(a.x * cs0.x - b.x * cs0.y, a.y * cs0.z - b.y * cs0.w,
                                                 a.z * cs1.x - b.z * cs1.y, a.w * cs1.z - b.w * cs1.w));
      store4(q + (size_t)r * d + c1, make_float4(b.x * cs0.x + a.x * cs0.y, b.y * cs0.z + a.y * cs0.w,
                                                 b.z * cs1.x + a.z * cs1.y, b.w * cs1.z + a.w * cs1.w));
    }
    if (store) {
      float4 a = sum_partials4(P, r, d + c0), b = sum_partials4(P, r, d + c1);
      a.x *= sc; a.y *= sc; a.z *= sc; a.w *= sc; b.x *= sc; b.y *= sc; b.z *= sc; b.w *= sc;
      const size_t o = ((size_t)h * max_ctx + slot) * dh + i;
      store4(kc + o, make_float4(a.x * cs0.x - b.x * cs0.y, a.y * cs0.z - b.y * cs0.w,
                                 a.z * cs1.x - b.z * cs1.y, a.w * cs1.z - b.w * cs1.w));
      store4(kc + o + half, make_float4(b.x * cs0.x + a.x * cs0.y, b.y * cs0.z + a.y * cs0.w,
                                        b.z * cs1.x + a.z * cs1.y, b.w * cs1.z + a.w * cs1.w));
      float4 v0 = sum_partials4(P, r, 2 * d + c0), v1 = sum_partials4(P, r, 2 * d + c1);
      store4(vc + o, make_float4(v0.x * sc, v0.y * sc, v0.z * sc, v0.w * sc));
      store4(vc + o + half, make_float4(v1.x * sc, v1.y * sc, v1.z * sc, v1.w * sc));
    }
  }
}

// The same for G row groups in one launch (blockIdx.z = group): group g's rows start at row g * rpg of P, q and rs and
// use their own row table, rotary table and cache.
template <typename T>
__global__ void __launch_bounds__(256)
qkv_rope_groups_kernel(PartialView P, RopeGroups gr, T* __restrict__ q, int n_heads, int dh, int max_ctx, RowScale rs) {
  pdl_wait();
  pdl_launch_dependents();
  const int g = blockIdx.z, rl = blockIdx.x, r = g * gr.rpg + rl;
  const RowMeta* meta = gr.meta[g];
  const float2* rope = gr.rope[g];
  T* kc = (T*)gr.kc[g];
  T* vc = (T*)gr.vc[g];
  const int half = dh >> 1, d = n_heads * dh, quads = half >> 2;
  const bool live = rl < meta->n_rows;
  const int slot = meta->slot[rl];
  const bool store = live && slot >= 0 && slot < max_ctx;
  const float sc = row_scale(rs, r);
  for (int idx = blockIdx.y * blockDim.x + threadIdx.x; idx < n_heads * quads; idx += gridDim.y * blockDim.x) {
    const int h = idx / quads, i = (idx - h * quads) * 4;
    const float4 cs0 = *reinterpret_cast<const float4*>(rope + rl * half + i);
    const float4 cs1 = *reinterpret_cast<const float4*>(rope + rl * half + i + 2);
    const int c0 = h * dh + i, c1 = c0 + half;
    {
      float4 a = sum_partials4(P, r, c0), b = sum_partials4(P, r, c1);
      a.x *= sc; a.y *= sc; a.z *= sc; a.w *= sc; b.x *= sc; b.y *= sc; b.z *= sc; b.w *= sc;
      store4(q + (size_t)r * d + c0, make_float4(a.x * cs0.x - b.x * cs0.y, a.y * cs0.z - b.y * cs0.w,
                                                 a.z * cs1.x - b.z * cs1.y, a.w * cs1.z - b.w * cs1.w));
      store4(q + (size_t)r * d + c1, make_float4(b.x * cs0.x + a.x * cs0.y, b.y * cs0.z + a.y * cs0.w,
                                                 b.z * cs1.x + a.z * cs1.y, b.w * cs1.z + a.w * cs1.w));
    }
    if (store) {
      float4 a = sum_partials4(P, r, d + c0), b = sum_partials4(P, r, d + c1);
      a.x *= sc; a.y *= sc; a.z *= sc; a.w *= sc; b.x *= sc; b.y *= sc; b.z *= sc; b.w *= sc;
      const size_t o = ((size_t)h * max_ctx + slot) * dh + i;
      store4(kc + o, make_float4(a.x * cs0.x - b.x * cs0.y, a.y * cs0.z - b.y * cs0.w,
                                 a.z * cs1.x - b.z * cs1.y, a.w * cs1.z - b.w * cs1.w));
      store4(kc + o + half, make_float4(b.x * cs0.x + a.x * cs0.y, b.y * cs0.z + a.y * cs0.w,
                                        b.z * cs1.x + a.z * cs1.y, b.w * cs1.z + a.w * cs1.w));
      float4 v0 = sum_partials4(P, r, 2 * d + c0), v1 = sum_partials4(P, r, 2 * d + c1);
      store4(vc + o, make_float4(v0.x * sc, v0.y * sc, v0.z * sc, v0.w * sc));
      store4(vc + o + half, make_float4(v1.x * sc, v1.y * sc, v1.z * sc, v1.w * sc));
    }
  }
}

void launch_qkv_rope_groups(PartialView P, const RopeGroups& gr, void* q, int dtype, int n_heads, int head_dim, int max_ctx,
                            cudaStream_t st, RowScale rs) {
  const int items = n_heads * head_dim / 8;
  const int threads = items >= 128 ? 128 : (items + 31) / 32 * 32;
  const int gy = (items + threads - 1) / threads;
  AMPH_DISPATCH(dtype, launch_pdl(qkv_rope_groups_kernel<T>, dim3(gr.rpg, gy, gr.G), dim3(threads), 0, st, P, gr, (T*)q, n_heads,
                                  head_dim, max_ctx, rs));
}

void launch_qkv_rope(PartialView P, const RowMeta* meta, const float2* rope, void* q, KvView kv, int dtype,
                     int rows, int n_heads, int head_dim, int max_ctx, cudaStream_t st, RowScale rs) {
  const int items = n_heads * head_dim / 8;
  const int threads = items >= 128 ? 128 : (items + 31) / 32 * 32;
  const int gy = (items + threads - 1) / threads;
  AMPH_DISPATCH(dtype, launch_pdl(qkv_rope_kernel<T>, dim3(rows, gy), dim3(threads), 0, st, P, meta, rope, (T*)q,
                                  (T*)kv.k, (T*)kv.v, n_heads, head_dim, max_ctx, rs));
}

// --------------------------------------------------------------------------------------------
// Tree attention on CUDA cores (fp32 caches), split over the KV axis (flash-decoding form), with the tree as a bitmask.
// Grid (head, split, row block of 16).  Slots below meta->base are visible to every row; slot base + m is visible to row r iff
// bit m of mask[r] is set.  Sixteen threads share a row: four keys of a tile each for the scores, a sixteenth of the head
// dimension each for the output.  Bound: latency (one L2 round trip per 64 keys, all of a tile's loads in flight together).
// A single split writes the final rows itself.  At 16 rows and 70 keys 5.7 us; 64-row blocks (mostly empty) with 32-key tiles
// fetched four bytes at a time, and a merge launch always, took 15.
// --------------------------------------------------------------------------------------------
constexpr int kAttRows = 16;     // query rows per block
constexpr int kAttTile = 64;     // keys per inner tile
constexpr int kAttThreads = 256;

template <typename T, int DH>
__global__ void __launch_bounds__(kAttThreads)
tree_attn_kernel(const T* __restrict__ q, const T* __restrict__ kc, const T* __restrict__ vc,
                 const RowMeta* __restrict__ meta, float* __restrict__ po, float* __restrict__ pml, T* __restrict__ out,
                 int rows_cap, int n_heads, int max_ctx) {
  pdl_wait();
  pdl_launch_dependents();
  constexpr int QS = DH + 4;                       // padded row strides (bank-conflict free float4 reads)
  constexpr int SEG = DH / 16;                     // output dims owned by one thread
  constexpr int KEYS = kAttTile / 16;              // keys of a tile per thread
  extern __shared__ __align__(16) float sm[];
  float* Qs = sm;                                  // [16][QS]
  float* Ks = Qs + kAttRows * QS;                  // [64][QS]
  float* Vs = Ks + kAttTile * QS;                  // [64][DH]
  float* Ss = Vs + kAttTile * DH;                  // [16][65]
  const int h = blockIdx.x, split = blockIdx.y, tid = threadIdx.x;
  const int r = tid >> 4, l16 = tid & 15;
  const int rg = blockIdx.z * kAttRows + r;        // global row
  const int base = meta->base, n_rows = meta->n_rows;
  const int d = n_heads * DH;
  const int total = base + n_rows;                 // slots that can be visible
  int chunk = (total + gridDim.y - 1) / gridDim.y;
  chunk = (chunk + kAttTile - 1) / kAttTile * kAttTile;
  const int s_lo = split * chunk;
  int s_hi = s_lo + chunk;
  if (s_hi > total) s_hi = total;
  if (s_hi > max_ctx) s_hi = max_ctx;
  const bool live = rg < n_rows;
  u64 m0 = 0, m1 = 0;
  if (live) { m0 = meta->mask[rg][0]; m1 = meta->mask[rg][1]; }
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i = tid; i < kAttRows * DH / 4; i += kAttThreads) {
    const int rr = i / (DH / 4), c = (i - rr * (DH / 4)) * 4, g = blockIdx.z * kAttRows + rr;
    store4(Qs + rr * QS + c, g < rows_cap ? load4(q + (size_t)g * d + h * DH + c) : zero);
  }
  float acc[SEG];
#pragma unroll
  for (int i = 0; i < SEG; ++i) acc[i] = 0.f;
  float mrun = -INFINITY, lrun = 0.f;
  const float scale = 1.0f / sqrtf((float)DH);
  const T* kh = kc + (size_t)h * max_ctx * DH;
  const T* vh = vc + (size_t)h * max_ctx * DH;
  for (int t0 = s_lo; t0 < s_hi; t0 += kAttTile) {
    constexpr int PER = kAttTile * DH / 4 / kAttThreads;
    float4 kr[PER], vr[PER];
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int e = tid + i * kAttThreads, j = e / (DH / 4), c = (e - j * (DH / 4)) * 4;
      const bool in_range = t0 + j < s_hi;
      kr[i] = in_range ? load4(kh + (size_t)(t0 + j) * DH + c) : zero;
      vr[i] = in_range ? load4(vh + (size_t)(t0 + j) * DH + c) : zero;
    }
    __syncthreads();                               // the previous tile has been read
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int e = tid + i * kAttThreads, j = e / (DH / 4), c = (e - j * (DH / 4)) * 4;
      store4(Ks + j * QS + c, kr[i]);
      store4(Vs + j * DH + c, vr[i]);
    }
    __syncthreads();
    float sc[KEYS];
#pragma unroll
    for (int jj = 0; jj < KEYS; ++jj) sc[jj] = 0.f;
    const float4* qa = reinterpret_cast<const float4*>(Qs + r * QS);
#pragma unroll 4
    for (int c = 0; c < DH / 4; ++c) {
      const float4 a = qa[c];
#pragma unroll
      for (int jj = 0; jj < KEYS; ++jj) {
        const float4 b = *reinterpret_cast<const float4*>(Ks + (jj * 16 + l16) * QS + 4 * c);
        sc[jj] += a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w;
      }
    }
    float tmax = -INFINITY;
#pragma unroll
    for (int jj = 0; jj < KEYS; ++jj) {
      const int s = t0 + jj * 16 + l16;
      bool vis = live && s < s_hi;
      if (vis && s >= base) {
        const int m = s - base;
        vis = m < 64 ? ((m0 >> m) & 1ull) : ((m1 >> (m - 64)) & 1ull);
      }
      sc[jj] = vis ? sc[jj] * scale : -INFINITY;
      tmax = fmaxf(tmax, sc[jj]);
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
    const float mnew = fmaxf(mrun, tmax);
    const bool any = mnew != -INFINITY;            // else nothing is visible yet for this row
    const float corr = any ? expf(mrun - mnew) : 1.f;      // exp(-inf) = 0 on the first visible tile
    float psum = 0.f;
#pragma unroll
    for (int jj = 0; jj < KEYS; ++jj) {
      const float p = any && sc[jj] != -INFINITY ? expf(sc[jj] - mnew) : 0.f;
      Ss[r * (kAttTile + 1) + jj * 16 + l16] = p;
      psum += p;
    }
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) psum += __shfl_xor_sync(0xffffffffu, psum, o);
    lrun = lrun * corr + psum;
    mrun = mnew;
    __syncwarp();                                  // a row's sixteen threads sit in one warp
#pragma unroll
    for (int i = 0; i < SEG; ++i) acc[i] *= corr;
#pragma unroll 4
    for (int j = 0; j < kAttTile; ++j) {
      const float p = Ss[r * (kAttTile + 1) + j];
#pragma unroll
      for (int c = 0; c < SEG; c += 4) {
        const float4 v = *reinterpret_cast<const float4*>(Vs + j * DH + l16 * SEG + c);
        acc[c] += p * v.x; acc[c + 1] += p * v.y; acc[c + 2] += p * v.z; acc[c + 3] += p * v.w;
      }
    }
  }
  if (rg >= rows_cap) return;
  if (out != nullptr) {
    const float inv = lrun > 0.f ? 1.0f / lrun : 0.f;
#pragma unroll
    for (int c = 0; c < SEG; c += 4)
      store4(out + (size_t)rg * d + h * DH + l16 * SEG + c, make_float4(acc[c] * inv, acc[c + 1] * inv, acc[c + 2] * inv, acc[c + 3] * inv));
    return;
  }
  const size_t o = (((size_t)split * n_heads + h) * rows_cap + rg);
#pragma unroll
  for (int c = 0; c < SEG; c += 4) store4(po + o * DH + l16 * SEG + c, make_float4(acc[c], acc[c + 1], acc[c + 2], acc[c + 3]));
  if (l16 == 0) { pml[o * 2] = mrun; pml[o * 2 + 1] = lrun; }
}

template <typename T>
__global__ void attn_combine_kernel(const float* __restrict__ po, const float* __restrict__ pml,
                                    T* __restrict__ out, int splits, int rows_cap, int n_heads, int dh, int early) {
  if (early) pdl_launch_dependents();
  pdl_wait();
  if (!early) pdl_launch_dependents();
  const int r = blockIdx.x, h = blockIdx.y;
  const size_t stride = (size_t)n_heads * rows_cap, o0 = (size_t)h * rows_cap + r;
  if (splits <= 16) {
    // every load of the launch is issued before the first use: (max, sum) of all splits, then the partial
    // outputs of all splits for this thread's column
    float2 ml[16];
#pragma unroll
    for (int s = 0; s < 16; ++s)
      ml[s] = s < splits ? *reinterpret_cast<const float2*>(pml + (o0 + s * stride) * 2) : make_float2(-INFINITY, 0.f);
    for (int c = threadIdx.x; c < dh; c += blockDim.x) {
      float v[16];
#pragma unroll
      for (int s = 0; s < 16; ++s) v[s] = s < splits ? po[(o0 + s * stride) * dh + c] : 0.f;
      float M = -INFINITY;
#pragma unroll
      for (int s = 0; s < 16; ++s) M = fmaxf(M, ml[s].x);
      float den = 0.f, num = 0.f;
#pragma unroll
      for (int s = 0; s < 16; ++s)
        if (ml[s].x != -INFINITY) {
          const float w = expf(ml[s].x - M);
          den += ml[s].y * w;
          num += v[s] * w;
        }
      out[(size_t)r * n_heads * dh + h * dh + c] = from_f<T>(den > 0.f ? num / den : 0.f);
    }
    return;
  }
  float M = -INFINITY;
  for (int s = 0; s < splits; ++s) M = fmaxf(M, pml[(o0 + s * stride) * 2]);
  float den = 0.f;
  for (int s = 0; s < splits; ++s) {
    const float m = pml[(o0 + s * stride) * 2];
    if (m != -INFINITY) den += pml[(o0 + s * stride) * 2 + 1] * expf(m - M);
  }
  for (int c = threadIdx.x; c < dh; c += blockDim.x) {
    float num = 0.f;
    for (int s = 0; s < splits; ++s) {
      const float m = pml[(o0 + s * stride) * 2];
      if (m != -INFINITY) num += po[(o0 + s * stride) * dh + c] * expf(m - M);
    }
    out[(size_t)r * n_heads * dh + h * dh + c] = from_f<T>(den > 0.f ? num / den : 0.f);
  }
}

template <typename T, int DH>
static void tree_attention_t(const void* q, KvView kv, const RowMeta* meta, AttnScratch sc, void* out,
                             int rows, int n_heads, int max_ctx, int splits, cudaStream_t st) {
  const size_t smem = sizeof(float) * (kAttRows * (DH + 4) + kAttTile * (DH + 4) + kAttTile * DH + kAttRows * (kAttTile + 1));
  cudaFuncSetAttribute(tree_attn_kernel<T, DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  launch_pdl(tree_attn_kernel<T, DH>, dim3(n_heads, splits, (rows + kAttRows - 1) / kAttRows), dim3(kAttThreads), smem, st, (const T*)q,
             (const T*)kv.k, (const T*)kv.v, meta, sc.o, sc.ml, splits == 1 ? (T*)out : (T*)nullptr, rows, n_heads, max_ctx);
  if (splits > 1)
    launch_pdl(attn_combine_kernel<T>, dim3(rows, n_heads), dim3(DH < 128 ? 64 : 128), 0, st, sc.o, sc.ml, (T*)out, splits, rows,
               n_heads, DH, 0);
}

void launch_attn_combine(AttnScratch sc, void* out, int dtype, int splits, int rows, int n_heads, int head_dim,
                         cudaStream_t st, int early) {
  AMPH_DISPATCH(dtype, launch_pdl(attn_combine_kernel<T>, dim3(dim3(rows, n_heads)), dim3(head_dim < 128 ? 64 : 128), 0, st, sc.o, sc.ml,
                                  (T*)out, splits, rows, n_heads, head_dim, early));
}

void launch_tree_attention(const void* q, KvView kv, const RowMeta* meta, AttnScratch sc, void* out, int dtype,
                           int rows, int n_heads, int head_dim, int max_ctx, int ctx_hi, int max_splits,
                           cudaStream_t st, int early, int separate_merge) {
  int splits = (ctx_hi + 127) / 128;
  if (splits > max_splits) splits = max_splits;
  if (splits < 1) splits = 1;
  if (dtype == AMPH_DTYPE_BF16) {                    // tensor-core path; the kernel below serves fp32 caches
    if (launch_tree_attention_mma(q, kv, meta, sc, rows, n_heads, head_dim, max_ctx, splits, st,
                                  separate_merge ? nullptr : out))
      return;
    launch_pdl(attn_combine_kernel<bf16>, dim3(dim3(rows, n_heads)), dim3(head_dim < 128 ? 64 : 128), 0, st, sc.o, sc.ml, (bf16*)out, splits,
                                                                                        rows, n_heads, head_dim, early);
    return;
  }
  if (head_dim == 64) {
    AMPH_DISPATCH(dtype, (tree_attention_t<T, 64>(q, kv, meta, sc, out, rows, n_heads, max_ctx, splits, st)));
  } else {
    AMPH_DISPATCH(dtype, (tree_attention_t<T, 128>(q, kv, meta, sc, out, rows, n_heads, max_ctx, splits, st)));
  }
}

// --------------------------------------------------------------------------------------------
// SwiGLU on the fused gate / up projection: act = silu(gate) * up
// --------------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256)
swiglu_kernel(PartialView P, T* __restrict__ act, int rows, int f, RowScale rs, int early) {
  if (early) pdl_launch_dependents();
  pdl_wait();
  if (!early) pdl_launch_dependents();
  const int r = blockIdx.x;
  const float sc = row_scale(rs, r);
  for (int c = (blockIdx.y * blockDim.x + threadIdx.x) * 4; c < f; c += gridDim.y * blockDim.x * 4) {
    const float4 g = sum_partials4(P, r, c), u = sum_partials4(P, r, f + c);
    float4 o;
    float t;
    t = g.x * sc; o.x = t / (1.0f + expf(-t)) * (u.x * sc);
    t = g.y * sc; o.y = t / (1.0f + expf(-t)) * (u.y * sc);
    t = g.z * sc; o.z = t / (1.0f + expf(-t)) * (u.z * sc);
    t = g.w * sc; o.w = t / (1.0f + expf(-t)) * (u.w * sc);
    store4(act + (size_t)r * f + c, o);
  }
}

void launch_swiglu(PartialView P, void* act, int dtype, int rows, int f, cudaStream_t st, RowScale rs, int early) {
  int gy = (f / 4 + 255) / 256;
  if (gy > 16) gy = 16;
  AMPH_DISPATCH(dtype, launch_pdl(swiglu_kernel<T>, dim3(rows, gy), dim3(256), 0, st, P, (T*)act, rows, f, rs, early));
}

// --------------------------------------------------------------------------------------------
// Plain projection kernel, fp32 accumulate: fp32 models, shapes the tensor-core kernel does not cover, and its A/B check.
// Grid (8 * O features, weight matrix, R rows).  A warp owns O features and all R rows of its block: weights straight to
// registers, each lane 32 bytes of 1 KB of the row, fetched before the dependency wait and one chunk ahead after it;
// activations through shared memory (cp.async, two buffers), so the block's eight warps read them from L2 once.
// Bound: latency at the sizes fp32 models are run at (16 rows, 256 columns: 2.7 us of the chain; with one launch per weight
// matrix, activations read by every warp for itself and weights again for every eight rows: 7.3 us a launch).
// --------------------------------------------------------------------------------------------
template <typename T> struct Vec16;
template <> struct Vec16<float> { static constexpr int N = 4; };
template <> struct Vec16<bf16> { static constexpr int N = 8; };

template <typename T>
__device__ __forceinline__ void unpack16(const uint4& v, float* out);
template <>
__device__ __forceinline__ void unpack16<float>(const uint4& v, float* out) {
  out[0] = __uint_as_float(v.x); out[1] = __uint_as_float(v.y); out[2] = __uint_as_float(v.z); out[3] = __uint_as_float(v.w);
}
template <>
__device__ __forceinline__ void unpack16<bf16>(const uint4& v, float* out) {
  const unsigned w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    out[2 * i] = __uint_as_float(w[i] << 16);
    out[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool live) {      // zeros where !live
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "r"(live ? 16 : 0)
               : "memory");
}

// row_scale shared by the 16 lanes of a half warp (all of them call; rows beyond `rows`: 1); t: the lane's first entry
__device__ __forceinline__ float row_scale16(const RowScale& rs, int row, int rows, float t) {
  if (rs.ss == nullptr) return 1.0f;
  if (row < rows)
    for (int c = 16 + (threadIdx.x & 15); c < rs.chunks; c += 16) t += rs.ss[(size_t)row * rs.chunks + c];
#pragma unroll
  for (int m = 8; m > 0; m >>= 1) t += __shfl_xor_sync(0xffffffffu, t, m);
  return row < rows ? 1.0f / sqrtf(t / (float)rs.d + rs.eps) : 1.0f;
}

struct GemmSegs { GemmSeg s[kMaxK]; };
constexpr int kPlainThreads = 256;
constexpr int kPlainChunk = 1024;        // bytes of a row per step: two 16-byte loads per lane
constexpr int kPlainOneFeature = 296;    // blocks (two per SM) up to which a warp has one feature: see launch_gemm_generic

// What becomes of the sums (16-row blocks of fp32 models; PLAIN: they go to P).  A launch per layer and step saved for each of the
// others: in a 2-layer model of width 256 rotary embedding 2.1 us of the chain, SwiGLU 1.9, each residual update 1.4.
//   SWIGLU: O = 2, a warp has a feature's gate and up row;  ROPE: O = 2, both members of a rotation pair, blockIdx.y = q, k, v;
//   RESID: O = 1, x += sum, xn = gain * x, and the eight features' squares of a row meet in shared memory (ss[row][block]).
// SWIGLU and ROPE let the next kernel start only by ending.  Its blocks would be placed beside theirs, on the few SMs with room, and
// stay there: attention right behind ROPE took 24.8 us instead of 8.9 (width 256, 64 rows), the down projection behind SWIGLU lost
// its spread too.  RESID triggers at once: what follows it starts with weights that wait for nothing.
// Us a step of an 8-layer model with separate kernels / with these forms: width 256, 16 rows 252 / 212, 512 rows 1338 / 1174; width
// 512 402 / 369 and 2451 / 2406; width 1024 692 / 621 and 6167 / 6035; width 2048 1499 / 1331 and 19000 / 18337.
enum { PLAIN_P = 0, PLAIN_SWIGLU = 1, PLAIN_ROPE = 2, PLAIN_RESID = 3 };
struct PlainEpi {
  RowScale rs;              // SWIGLU, ROPE: deferred division of the activation rows
  void* dst;                // SWIGLU: act [rows][out]; ROPE: q [rows][d]; RESID: xn [rows][out]
  RopeGroups gr;            // ROPE
  float inv_rpg;            // ROPE: 1 / gr.rpg
  int dh, max_ctx;
  float* x;                 // RESID [rows][out]
  const void* gain;         // RESID: or NULL (x only)
  float* ss;
};

template <typename T, int R, int O, int EPI>
__global__ void __launch_bounds__(kPlainThreads)
gemm_generic_kernel(const T* __restrict__ X, int ldx, const __grid_constant__ GemmSegs segs, int out, int in, float* __restrict__ P, int ldp, int rows,
                    int wait_first, const __grid_constant__ PlainEpi epi) {
  if (EPI == PLAIN_P || EPI == PLAIN_RESID) pdl_launch_dependents();
  constexpr int V = Vec16<T>::N, KC = kPlainChunk / (int)sizeof(T);
  __shared__ __align__(16) uint4 xs[2][R][kPlainChunk / 16];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int item = blockIdx.x * (kPlainThreads / 32) + warp, r0 = blockIdx.z * R;
  // first feature of this warp, the distance of its others, and their matrix
  const int half = EPI == PLAIN_ROPE ? epi.dh >> 1 : 0;          // a power of two
  const int o0 = EPI == PLAIN_ROPE ? 2 * (item & -half) + (item & (half - 1)) : EPI == PLAIN_SWIGLU ? item : item * O;
  const int step = EPI == PLAIN_ROPE ? half : EPI == PLAIN_SWIGLU ? 0 : 1;
  auto weights = [&](int i) { return (const T*)segs.s[EPI == PLAIN_SWIGLU ? i : blockIdx.y].w; };
  const int chunks = (in + KC - 1) / KC;
  uint4 w[O][2];
  auto load_w = [&](int c) {
#pragma unroll
    for (int i = 0; i < O; ++i)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int k = c * KC + (v * 32 + lane) * V;
        w[i][v] = make_uint4(0u, 0u, 0u, 0u);
        if (o0 + i * step < out && k < in) w[i][v] = *reinterpret_cast<const uint4*>(weights(i) + (size_t)(o0 + i * step) * in + k);
      }
  };
  auto load_x = [&](int c) {
    for (int i = threadIdx.x; i < R * (kPlainChunk / 16); i += kPlainThreads) {
      const int r = i / (kPlainChunk / 16), j = i - r * (kPlainChunk / 16), k = c * KC + j * V;
      const bool live = r0 + r < rows && k < in;
      cp_async16(&xs[c & 1][r][j], live ? X + (size_t)(r0 + r) * ldx + k : X, live);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (wait_first) pdl_wait();
  load_w(0);
  pdl_wait();
  auto group_of = [&](int r) { return (int)(((float)r + 0.5f) * epi.inv_rpg); };       // r / rpg: both are below 2^10
  // the row that this lane ends up with
  constexpr int same = R <= 32 ? 32 / R : 1;             // lanes that end up with the same row
  auto own_row = [&] {
    int row = 0;
#pragma unroll
    for (int h = R / 2, m = 16; h > 0; h >>= 1, m >>= 1) row += (lane & m) ? h : 0;
    return row;
  };
  constexpr bool SCALED = EPI == PLAIN_SWIGLU || EPI == PLAIN_ROPE;
  __shared__ float inv_s[SCALED ? R : 1];                // 1 / rms of the block's rows, from 16 lanes each
  static_assert(!SCALED || R * 16 == kPlainThreads, "16 lanes a row");
  // What the epilogue reads is asked for ahead of the activations and looked at behind the main loop's first loads, or its end: a
  // stall ahead of them is added to every block (512 rows at width 512, gate / up 91 us, now 85; q / k / v 56 and 51).
  float old = 0.f, ss0 = 0.f;
  float2 cs = make_float2(1.f, 0.f);
  int slot = -1, live = 0;
  if (EPI != PLAIN_P) {
    const int rg = r0 + own_row(), rs = r0 + (int)(threadIdx.x >> 4);
    if (SCALED && epi.rs.ss != nullptr && rs < rows && (threadIdx.x & 15) < epi.rs.chunks) ss0 = epi.rs.ss[rs * epi.rs.chunks + (threadIdx.x & 15)];
    if (EPI == PLAIN_RESID && rg < rows && o0 < out) old = epi.x[(size_t)rg * out + o0];
    if (EPI == PLAIN_ROPE && rg < rows && o0 < out) {
      const int g = group_of(rg), rl = rg - g * epi.gr.rpg;
      if (blockIdx.y < 2) cs = epi.gr.rope[g][(size_t)rl * half + (o0 & (half - 1))];
      if (blockIdx.y > 0) { slot = epi.gr.meta[g]->slot[rl]; live = epi.gr.meta[g]->n_rows; }
    }
  }
  load_x(0);
  float acc[O][R];
#pragma unroll
  for (int i = 0; i < O; ++i)
#pragma unroll
    for (int r = 0; r < R; ++r) acc[i][r] = 0.f;
  for (int c = 0; c < chunks; ++c) {
    float wv[O][2][V];
#pragma unroll
    for (int i = 0; i < O; ++i)
#pragma unroll
      for (int v = 0; v < 2; ++v) unpack16<T>(w[i][v], wv[i][v]);
    if (c + 1 < chunks) {
      load_x(c + 1);
      load_w(c + 1);
    }
    if (SCALED && c == 0) {
      const float inv = row_scale16(epi.rs, r0 + (int)(threadIdx.x >> 4), rows, ss0);
      if ((threadIdx.x & 15) == 0) inv_s[threadIdx.x >> 4] = inv;
    }
    if (c + 1 < chunks) asm volatile("cp.async.wait_group 1;" ::: "memory");
    else asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        float xv[V];
        unpack16<T>(xs[c & 1][r][v * 32 + lane], xv);
#pragma unroll
        for (int i = 0; i < O; ++i)
#pragma unroll
          for (int e = 0; e < V; ++e) acc[i][r] += wv[i][v][e] * xv[e];
      }
    __syncthreads();
  }
  // sums over the lanes: at every step a lane keeps half of its rows and hands the other half to its partner
#pragma unroll
  for (int i = 0; i < O; ++i) {
#pragma unroll
    for (int h = R / 2, m = 16; m > 0; h >>= 1, m >>= 1) {
      if (h > 0) {
        const bool up = (lane & m) != 0;
#pragma unroll
        for (int r = 0; r < h; ++r) {
          const float give = up ? acc[i][r] : acc[i][r + h], keep = up ? acc[i][r + h] : acc[i][r];
          acc[i][r] = keep + __shfl_xor_sync(0xffffffffu, give, m);
        }
      } else {
        acc[i][0] += __shfl_xor_sync(0xffffffffu, acc[i][0], m);
      }
    }
    if constexpr (EPI == PLAIN_P) {
      const int rg = r0 + own_row();
      if (lane % same == 0 && rg < rows && o0 + i < out) P[(size_t)rg * ldp + blockIdx.y * out + o0 + i] = acc[i][0];
    }
  }
  const int row = own_row(), rg = r0 + row;
  const bool mine = lane % same == 0 && rg < rows && o0 < out;
  if constexpr (EPI == PLAIN_SWIGLU) {
    const float scale = inv_s[row], t = acc[0][0] * scale;
    if (mine) ((T*)epi.dst)[(size_t)rg * out + o0] = from_f<T>(t / (1.0f + expf(-t)) * (acc[1][0] * scale));
  } else if constexpr (EPI == PLAIN_ROPE) {
    const float scale = inv_s[row], a = acc[0][0] * scale, b = acc[1][0] * scale;
    if (!mine) return;
    T* dst = (T*)epi.dst + (size_t)rg * out + o0;
    if (blockIdx.y > 0) {
      const int g = group_of(rg), i = o0 & (half - 1);
      if (rg - g * epi.gr.rpg >= live || slot < 0 || slot >= epi.max_ctx) return;
      // head o0 / dh
      dst = (T*)(blockIdx.y == 1 ? epi.gr.kc[g] : epi.gr.vc[g]) + (size_t)(o0 - i) * epi.max_ctx + (size_t)slot * epi.dh + i;
    }
    dst[0] = from_f<T>(blockIdx.y < 2 ? a * cs.x - b * cs.y : a);
    dst[half] = from_f<T>(blockIdx.y < 2 ? b * cs.x + a * cs.y : b);
  } else if constexpr (EPI == PLAIN_RESID) {
    __shared__ float sq[kPlainThreads / 32][R];
    const float v = acc[0][0] + old;
    if (mine) {
      epi.x[(size_t)rg * out + o0] = v;
      if (epi.gain != nullptr) ((T*)epi.dst)[(size_t)rg * out + o0] = from_f<T>(to_f(((const T*)epi.gain)[o0]) * v);
    }
    if (epi.gain == nullptr) return;
    if (lane % same == 0) sq[warp][row] = mine ? v * v : 0.f;
    __syncthreads();
    if (threadIdx.x < R && r0 + (int)threadIdx.x < rows) {
      float t = 0.f;
#pragma unroll
      for (int i = 0; i < kPlainThreads / 32; ++i) t += sq[i][threadIdx.x];
      epi.ss[(size_t)(r0 + threadIdx.x) * gridDim.x + blockIdx.x] = t;
    }
  }
}

// R = 4 for the drafting heads' few rows, 8 for theirs in a batch of two, else 16 (the rows a block does not have cost it as much
// as those it has: 5 to 8 rows in blocks of 16 took 70 us at 11008 x 4096 in bf16, now 41; 102 at 3 x 4096 x 4096 in fp32, now 73); two
// features a warp (half of the shared-memory reads) once one feature a warp gives more than two blocks per SM (8 rows: 51 us and
// 82 us with one).
void launch_gemm_generic(const void* x, int ldx, const GemmSeg* segs, int n_seg, int out, int in, float* P,
                         int ldp, int rows, int dtype, cudaStream_t st, int wait_first) {
  GemmSegs gs;
  for (int s = 0; s < kMaxK; ++s) gs.s[s].w = s < n_seg ? segs[s].w : nullptr;
  const int blocks = (out + 7) / 8;
  auto run = [&](auto kernel, int R, int O, auto* X) {
    launch_pdl(kernel, dim3((out + 8 * O - 1) / (8 * O), n_seg, (rows + R - 1) / R), dim3(kPlainThreads), 0, st, X, ldx, gs, out, in, P, ldp,
               rows, wait_first, PlainEpi());
  };
  AMPH_DISPATCH(dtype, const T* X = (const T*)x;
                if (rows <= 4) run(gemm_generic_kernel<T, 4, 1, PLAIN_P>, 4, 1, X);
                else if (rows <= 8 && blocks * n_seg <= kPlainOneFeature) run(gemm_generic_kernel<T, 8, 1, PLAIN_P>, 8, 1, X);
                else if (rows <= 8) run(gemm_generic_kernel<T, 8, 2, PLAIN_P>, 8, 2, X);
                else if ((long long)blocks * n_seg * ((rows + 15) / 16) <= kPlainOneFeature) run(gemm_generic_kernel<T, 16, 1, PLAIN_P>, 16, 1, X);
                else run(gemm_generic_kernel<T, 16, 2, PLAIN_P>, 16, 2, X));
}

// The fused forms, fp32: 16-row blocks, eight features (pairs) a block.  RESID only where launch_gemm_generic would take one feature a
// warp too: beyond that its blocks stage the activation rows twice as often as those of two features (256 rows at width 1024: 4716 us a
// prefill with it everywhere, 3350 with this rule, 3521 with no fused form).
static void plain_fused(void (*kernel)(const float*, int, GemmSegs, int, int, float*, int, int, int, PlainEpi), const void* x, const void* const* w,
                        int n_w, int items, int ny, int out, int in, int rows, const PlainEpi& epi, cudaStream_t st) {
  GemmSegs gs;
  for (int s = 0; s < kMaxK; ++s) gs.s[s].w = s < n_w ? w[s] : nullptr;
  launch_pdl(kernel, dim3((items + 7) / 8, ny, (rows + 15) / 16), dim3(kPlainThreads), 0, st, (const float*)x, in, gs, out, in, (float*)nullptr, 0,
             rows, 0, epi);
}

void launch_plain_swiglu(const void* x, const void* w_gate, const void* w_up, int f, int in, int rows, void* act, const RowScale& rs,
                         cudaStream_t st) {
  const void* w[2] = {w_gate, w_up};
  PlainEpi e = {};
  e.rs = rs;
  e.dst = act;
  plain_fused(gemm_generic_kernel<float, 16, 2, PLAIN_SWIGLU>, x, w, 2, f, 1, f, in, rows, e, st);
}

void launch_plain_qkv_rope(const void* x, const void* const* w, int d, int dh, int in, int rows, void* q, const RopeGroups& gr, int max_ctx,
                           const RowScale& rs, cudaStream_t st) {
  PlainEpi e = {};
  e.rs = rs;
  e.dst = q;
  e.gr = gr;
  e.inv_rpg = 1.0f / (float)gr.rpg;
  e.dh = dh;
  e.max_ctx = max_ctx;
  plain_fused(gemm_generic_kernel<float, 16, 2, PLAIN_ROPE>, x, w, 3, d / 2, 3, d, in, rows, e, st);
}

bool plain_resid_pays(int out, int rows) {
  return out <= kPlainResidMax && (long long)((out + 7) / 8) * ((rows + 15) / 16) <= kPlainOneFeature;
}

void launch_plain_resid(const void* x_in, const void* w, int out, int in, int rows, float* x, const void* gain, void* xn, float* ss,
                        cudaStream_t st) {
  PlainEpi e = {};
  e.dst = xn;
  e.x = x;
  e.gain = gain;
  e.ss = ss;
  plain_fused(gemm_generic_kernel<float, 16, 1, PLAIN_RESID>, x_in, &w, 1, out, 1, out, in, rows, e, st);
}

// --------------------------------------------------------------------------------------------
// draft module: last-row gather, head MLP epilogue (Eq. 2-4), fused K x K attention (Eq. 5)
// --------------------------------------------------------------------------------------------
// Rows 2 b, 2 b + 1 of `last`: the last pending row of each stage of sequence b (blockIdx.z), whose rows_per rows start at row
// b * rows_per of h1 / h2.
template <typename T>
__global__ void gather_last_kernel(const float* __restrict__ h1, const float* __restrict__ h2, int rows_per,
                                   const char* __restrict__ state, size_t state_stride, char* __restrict__ last, size_t last_stride,
                                   T* __restrict__ last_act, int d) {
  pdl_wait();
  pdl_launch_dependents();
  const int b = blockIdx.z;
  int lr = reinterpret_cast<const DevState*>(state + state_stride * b)->n_pending - 1;
  lr = lr < 0 ? 0 : (lr >= kPendMax ? kPendMax - 1 : lr);
  const float* src = (blockIdx.x == 0 ? h1 : h2) + ((size_t)b * rows_per + lr) * d;
  float* dst = reinterpret_cast<float*>(last + last_stride * b) + (size_t)blockIdx.x * d;
  T* act = last_act + ((size_t)b * 2 + blockIdx.x) * d;
  for (int c = (blockIdx.y * blockDim.x + threadIdx.x) * 4; c < d; c += gridDim.y * blockDim.x * 4) {
    const float4 v = load4(src + c);
    store4(dst + c, v);
    store4(act + c, v);
  }
}

void launch_gather_last(const float* h1, const float* h2, int rows_per, const void* state, size_t state_stride, void* last,
                        size_t last_stride, void* last_act, int dtype, int d, int batch, cudaStream_t st) {
  const int gy = (d / 4 + 255) / 256;
  AMPH_DISPATCH(dtype, launch_pdl(gather_last_kernel<T>, dim3(2, gy, batch), dim3(256), 0, st, h1, h2, rows_per, (const char*)state,
                                  state_stride, (char*)last, last_stride, (T*)last_act, d));
}

template <typename T>
__global__ void gather_diag_kernel(PartialView P, T* __restrict__ out, int K, int r) {
  pdl_wait();
  pdl_launch_dependents();
  const int row = blockIdx.x, k = row % K;
  for (int j = threadIdx.x; j < r; j += blockDim.x) out[(size_t)row * r + j] = from_f<T>(sum_partials(P, row, k * r + j));
}

void launch_gather_diag(PartialView P, void* out_act, int dtype, int K, int r, int batch, cudaStream_t st) {
  AMPH_DISPATCH(dtype, launch_pdl(gather_diag_kernel<T>, dim3(K * batch), dim3(256), 0, st, P, (T*)out_act, K, r));
}

struct BiasPtrs { const void* b[kMaxK]; };

template <typename T>
__global__ void mlp_heads_kernel(PartialView P, const char* __restrict__ last, size_t last_stride, BiasPtrs bias,
                                 const T* __restrict__ pe, float* __restrict__ hp, int hp_rows, float* __restrict__ ao,
                                 T* __restrict__ ao_act, int K, int n_sal, int d) {
  pdl_wait();
  pdl_launch_dependents();
  const int k = blockIdx.x, s = blockIdx.z;                 // head, sequence
  const int row = (k < K / 2 || n_sal == 1) ? 0 : 1;       // Eq. 2: first half of the heads <- stage 1
  const T* b = (const T*)bias.b[k];
  const float* src = reinterpret_cast<const float*>(last + last_stride * s) + (size_t)row * d;
  for (int c = (blockIdx.y * blockDim.x + threadIdx.x) * 4; c < d; c += gridDim.y * blockDim.x * 4) {
    const float4 w = sum_partials4(P, 2 * s + row, k * d + c), bb = load4(b + c), l = load4(src + c), e = load4(pe + (size_t)k * d + c);
    float4 v;
    float pre;
    pre = w.x + bb.x; v.x = l.x + pre / (1.0f + expf(-pre)) + e.x;
    pre = w.y + bb.y; v.y = l.y + pre / (1.0f + expf(-pre)) + e.y;
    pre = w.z + bb.z; v.z = l.z + pre / (1.0f + expf(-pre)) + e.z;
    pre = w.w + bb.w; v.w = l.w + pre / (1.0f + expf(-pre)) + e.w;
    store4(hp + ((size_t)s * hp_rows + k) * d + c, v);
    store4(ao + ((size_t)s * K + k) * d + c, v);          // the attention block updates this copy in place
    store4(ao_act + ((size_t)s * K + k) * d + c, v);
  }
}

void launch_mlp_heads(PartialView P, const void* last, size_t last_stride, const void* const* bias, const void* pe, float* hp, int hp_rows,
                      float* ao, void* ao_act, int dtype, int K, int n_sal, int d, int batch, cudaStream_t st) {
  BiasPtrs bp;
  for (int k = 0; k < kMaxK; ++k) bp.b[k] = k < K ? bias[k] : nullptr;
  const int gy = (d / 4 + 127) / 128;
  AMPH_DISPATCH(dtype, launch_pdl(mlp_heads_kernel<T>, dim3(K, gy, batch), dim3(128), 0, st, P, (const char*)last, last_stride, bp,
                                  (const T*)pe, hp, hp_rows, ao, (T*)ao_act, K, n_sal, d));
}

// One block per attention head and sequence (blockIdx.y: its K rows attend to each other only): the K x K score matrix,
// softmax and mixing stay in shared memory.
template <typename T>
__global__ void aeb_attention_kernel(PartialView P, T* __restrict__ out, int K, int n_heads, int dh) {
  pdl_wait();
  pdl_launch_dependents();
  extern __shared__ __align__(16) float sm[];
  float* qs = sm;                 // [K][dh]
  float* ks = qs + K * dh;
  float* vs = ks + K * dh;
  float* pr = vs + K * dh;        // [K][K]
  const int h = blockIdx.x, row0 = blockIdx.y * K, d = n_heads * dh;
  const int per = K * dh / 4;                            // float4 items per q / k / v block
  for (int i = threadIdx.x; i < 3 * per; i += blockDim.x) {
    const int which = i / per, j = (i - which * per) * 4;
    const int r = j / dh, c = j - r * dh;
    store4(sm + which * K * dh + j, sum_partials4(P, row0 + r, which * d + h * dh + c));
  }
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int p = w; p < K * K; p += nw) {               // one warp per (i, j) score
    const int i = p / K, j = p - i * K;
    float dot = 0.f;
    for (int c = lane; c < dh; c += 32) dot += qs[i * dh + c] * ks[j * dh + c];
    for (int s = 16; s > 0; s >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, s);
    if (lane == 0) pr[p] = dot / sqrtf((float)dh);
  }
  __syncthreads();
  if (threadIdx.x < K) {                              // bi-directional: every row sees every row
    const int i = threadIdx.x;
    float m = -INFINITY;
    for (int j = 0; j < K; ++j) m = fmaxf(m, pr[i * K + j]);
    float sum = 0.f;
    for (int j = 0; j < K; ++j) { const float e = expf(pr[i * K + j] - m); pr[i * K + j] = e; sum += e; }
    for (int j = 0; j < K; ++j) pr[i * K + j] /= sum;
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < K * dh; idx += blockDim.x) {
    const int i = idx / dh, c = idx - i * dh;
    float acc = 0.f;
    for (int j = 0; j < K; ++j) acc += pr[i * K + j] * vs[j * dh + c];
    out[(size_t)(row0 + i) * d + h * dh + c] = from_f<T>(acc);
  }
}

void launch_aeb_attention(PartialView P, void* out_act, int dtype, int K, int n_heads, int head_dim, int batch,
                          cudaStream_t st) {
  const size_t smem = sizeof(float) * (3 * K * head_dim + K * K);
  AMPH_DISPATCH(dtype, launch_pdl(aeb_attention_kernel<T>, dim3(n_heads, batch), dim3(128), smem, st, P, (T*)out_act, K, n_heads, head_dim));
}

// --------------------------------------------------------------------------------------------
// selection: top-k per drafting head (Eq. 6), greedy argmax per verified row
// order: value descending, equal values by ascending id
// --------------------------------------------------------------------------------------------
__device__ __forceinline__ bool better(float v, int i, float bv, int bi) {
  return v > bv || (v == bv && i < bi);
}

__device__ void block_best(float& v, int& i, float* sv, int* si) {
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, v, o);
    const int oi = __shfl_xor_sync(0xffffffffu, i, o);
    if (better(ov, oi, v, i)) { v = ov; i = oi; }
  }
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) { sv[w] = v; si[w] = i; }
  __syncthreads();
  v = sv[0]; i = si[0];
  for (int k = 1; k < nw; ++k)
    if (better(sv[k], si[k], v, i)) { v = sv[k]; i = si[k]; }
}

struct TopkCounts { int c[kMaxK]; };

// Selection keys: a larger key is a better candidate in the order above (-0 counts as +0); 0 is below every value and marks
// "nothing left", which is also what a NaN is: it compares with nothing, so it is nobody's candidate.
__device__ __forceinline__ uint32_t order_key(float v) {
  if (v != v) return 0u;
  const uint32_t u = __float_as_uint(v == 0.f ? 0.f : v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Stage 1: block (head k, chunk j, sequence b) reduces the split-K partials of its slice of the head's logits, stores them
// (debug tap) and selects the slice's own top-c_k; stage 2 (topk_tree_kernel) merges the slices' candidates.  The global
// top-c_k are each among their slice's top-c_k, so the result is the exact top-c_k of the row, in order.
// Every warp selects from an eighth of the slice (one warp-wide maximum and one minimum of ids per pick, no block barrier),
// then the first warp merges the eight sorted lists.  Bound: latency: picks made by the whole block, with two barriers each,
// and three launches per sequence cost a step 18 us more at 7B (32000 ids, 10 candidates) and 100 us more with eight sequences.
constexpr int kTopkChunks = kTopkCandChunks;
constexpr int kTopkThreads = 256;
constexpr int kTopkWarps = kTopkThreads / 32;

// One pick over the lanes of a warp: the best (key, lowest id) and the lane that holds it (-1: nothing left).
__device__ __forceinline__ int warp_pick(uint32_t key, int id, uint32_t& best_key, int& best_id) {
  best_key = __reduce_max_sync(0xffffffffu, key);
  best_id = (int)__reduce_min_sync(0xffffffffu, key == best_key ? (uint32_t)id : 0xffffffffu);
  const unsigned own = __ballot_sync(0xffffffffu, key == best_key && id == best_id);
  return best_key == 0u ? -1 : __ffs(own) - 1;
}

__global__ void __launch_bounds__(kTopkThreads)
topk_slice_kernel(PartialView P, int vocab, int chunk, int K, TopkCounts ck, char* __restrict__ cand, size_t cand_stride,
                  char* __restrict__ d_logits, size_t d_logits_stride, int vec) {
  pdl_wait();
  pdl_launch_dependents();
  extern __shared__ __align__(16) float slice[];
  __shared__ float2 lists[kTopkWarps][kTopkStride];
  const int k = blockIdx.x, j = blockIdx.y, b = blockIdx.z, row = b * K + k;
  const int lo = j * chunk, hi = lo + chunk < vocab ? lo + chunk : vocab;
  float* grow = reinterpret_cast<float*>(d_logits + d_logits_stride * b) + (size_t)k * vocab;
  for (int c = lo + threadIdx.x * 4; c < hi; c += blockDim.x * 4) {
    if (vec && c + 3 < hi) {
      const float4 v = sum_partials4(P, row, k * vocab + c);
      store4(grow + c, v);
      store4(slice + (c - lo), v);
    } else {
      for (int e = c; e < hi && e < c + 4; ++e) {
        const float v = sum_partials(P, row, k * vocab + e);
        grow[e] = v;
        slice[e - lo] = v;
      }
    }
  }
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, want = ck.c[k], n = hi - lo;
  const int part = (n + kTopkWarps - 1) / kTopkWarps, p0 = w * part, p1 = p0 + part < n ? p0 + part : n;
  // this lane's best entry strictly after the last pick it lost (its entries are p0 + lane, p0 + lane + 32, ...: ascending ids)
  uint32_t key = 0u, prev = 0xffffffffu;
  int id = 0x7fffffff, prev_id = -1;
  bool rescan = true;
  for (int t = 0; t < want; ++t) {
    if (rescan) {
      key = 0u;
      id = 0x7fffffff;
      for (int i = p0 + lane; i < p1; i += 32) {
        const uint32_t o = order_key(slice[i]);
        if (o > key && (o < prev || (o == prev && i > prev_id))) { key = o; id = i; }
      }
    }
    uint32_t bk;
    int bi;
    const int owner = warp_pick(key, id, bk, bi);
    if (lane == 0) lists[w][t] = owner < 0 ? make_float2(-INFINITY, __int_as_float(0x7fffffff)) : make_float2(slice[bi], __int_as_float(bi));
    rescan = lane == owner;
    if (rescan) { prev = bk; prev_id = bi; }
  }
  __syncthreads();
  if (w != 0) return;
  float2* out = reinterpret_cast<float2*>(cand + cand_stride * b) + ((size_t)k * gridDim.y + j) * kTopkStride;
  int at = 0;                                            // lane l < 8: next entry of warp l's sorted list
  for (int t = 0; t < want; ++t) {
    float2 e = make_float2(0.f, __int_as_float(0x7fffffff));
    if (lane < kTopkWarps && at < want) e = lists[lane][at];
    const int eid = __float_as_int(e.y);
    uint32_t bk;
    int bi;
    const int owner = warp_pick(eid == 0x7fffffff ? 0u : order_key(e.x), eid, bk, bi);
    if (owner < 0) { if (lane == 0) out[t] = make_float2(-INFINITY, __int_as_float(0x7fffffff)); continue; }
    if (lane == owner) { out[t] = make_float2(e.x, __int_as_float(lo + eid)); ++at; }
  }
}

// Node n of the verification pass of one sequence (Appendix A.1): tok[0] = root; tok[n] = head depth[n]'s candidate of
// rank rank[n]; optional overrides; row table: position C + depth, slot C + n, mask = ancestors (Fig. 5).
__device__ __forceinline__ void tree_row(const TreeDev* __restrict__ tree, const DevState* s, const int* topk_ids,
                                         const int* __restrict__ override_tok, int* __restrict__ tok, RowMeta* meta, int n) {
  const int N = tree->n_nodes, C = s->C;
  if (n == 0) { meta->base = C; meta->n_rows = N; }
  if (n < N) {
    if (n == 0) {
      tok[0] = s->root;
    } else {
      if (topk_ids) tok[n] = topk_ids[(tree->depth[n] - 1) * kTopkStride + tree->rank[n]];
      if (override_tok && override_tok[n] >= 0) tok[n] = override_tok[n];
    }
    meta->pos[n] = C + tree->depth[n];
    meta->slot[n] = C + n;
    meta->mask[n][0] = tree->anc[n][0];
    meta->mask[n][1] = tree->anc[n][1];
  } else {
    meta->pos[n] = C;
    meta->slot[n] = -1;
    meta->mask[n][0] = meta->mask[n][1] = 0ull;
  }
}

// Stage 2 and the candidate tree, one block per sequence: warp k merges head k's slice lists (lane j walks the sorted list of
// slice j), then the block lays the tree out from the merged candidates.
__global__ void __launch_bounds__(kTopkThreads)
topk_tree_kernel(const TopkTreeArgs a, int n_chunks, int K, TopkCounts ck) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ int ids_s[kMaxK * kTopkStride];
  const int b = blockIdx.x, k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (k < K) {
    const int want = ck.c[k];
    const float2* list = reinterpret_cast<const float2*>(a.cand + a.cand_stride * b) + ((size_t)k * n_chunks + lane) * kTopkStride;
    int* oid = reinterpret_cast<int*>(a.ids + a.ids_stride * b) + k * kTopkStride;
    float* oval = reinterpret_cast<float*>(a.vals + a.vals_stride * b) + k * kTopkStride;
    const float2 none = make_float2(0.f, __int_as_float(0x7fffffff));
    int at = 0;
    float2 e = lane < n_chunks ? list[0] : none, nx = lane < n_chunks && want > 1 ? list[1] : none;
    for (int t = 0; t < want; ++t) {
      const int eid = __float_as_int(e.y);
      uint32_t bk;
      int bi;
      const int owner = warp_pick(eid == 0x7fffffff ? 0u : order_key(e.x), eid, bk, bi);
      if (lane == (owner < 0 ? 0 : owner)) { oid[t] = bi; oval[t] = owner < 0 ? -INFINITY : e.x; ids_s[k * kTopkStride + t] = bi; }
      if (lane == owner) {                               // the entry after the next is fetched while the next one competes
        ++at;
        e = nx;
        nx = at + 1 < want ? list[at + 1] : none;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < kMaxRows)
    tree_row(a.tree, reinterpret_cast<const DevState*>(a.state + a.state_stride * b), ids_s, nullptr, a.tok + (size_t)b * a.rows,
             reinterpret_cast<RowMeta*>(a.meta + a.meta_stride * b), threadIdx.x);
}
static_assert(kTopkWarps >= kMaxK && kTopkChunks <= 32 && kTopkThreads >= kMaxRows, "a warp per head, a lane per slice, a thread per node");

void launch_topk_tree(PartialView P, int vocab, int K, const int* ck, const TopkTreeArgs& a, int batch, cudaStream_t st) {
  TopkCounts c;
  for (int k = 0; k < kMaxK; ++k) c.c[k] = k < K ? ck[k] : 0;
  const int vec = vocab % 4 == 0 && P.ld % 4 == 0;
  int chunk = (vocab + kTopkChunks - 1) / kTopkChunks;
  chunk = (chunk + 3) / 4 * 4;
  const int n_chunks = (vocab + chunk - 1) / chunk;
  const size_t bytes = (size_t)chunk * sizeof(float);
  if (bytes > 46 * 1024) cudaFuncSetAttribute(topk_slice_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  launch_pdl(topk_slice_kernel, dim3(K, n_chunks, batch), dim3(kTopkThreads), bytes, st, P, vocab, chunk, K, c, a.cand, a.cand_stride,
             a.d_logits, a.d_logits_stride, vec);
  launch_pdl(topk_tree_kernel, dim3(batch), dim3(kTopkThreads), 0, st, a, n_chunks, K, c);
}

// Greedy choice per verified row in two stages, like the top-k above: block (row, slice) reduces the partials of
// its slice of the row, stores the logits (debug tap) and its best (value, id); one thread per row then merges the
// slices (ties -> lowest id, the same order as a single pass).
constexpr int kArgmaxSlices = 8;

__global__ void __launch_bounds__(256)
argmax_slice_kernel(PartialView P, int vocab, int chunk, float2* __restrict__ cand, float* __restrict__ logits_out, int vec) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ float sv[32];
  __shared__ int si[32];
  const int r = blockIdx.x, j = blockIdx.y;
  const int lo = j * chunk, hi = lo + chunk < vocab ? lo + chunk : vocab;
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  for (int c = lo + threadIdx.x * 4; c < hi; c += blockDim.x * 4) {
    if (vec && c + 3 < hi) {
      const float4 v = sum_partials4(P, r, c);
      if (logits_out) store4(logits_out + (size_t)r * vocab + c, v);
      if (better(v.x, c, bv, bi)) { bv = v.x; bi = c; }
      if (better(v.y, c + 1, bv, bi)) { bv = v.y; bi = c + 1; }
      if (better(v.z, c + 2, bv, bi)) { bv = v.z; bi = c + 2; }
      if (better(v.w, c + 3, bv, bi)) { bv = v.w; bi = c + 3; }
    } else {
      for (int e = c; e < hi && e < c + 4; ++e) {
        const float v = sum_partials(P, r, e);
        if (logits_out) logits_out[(size_t)r * vocab + e] = v;
        if (better(v, e, bv, bi)) { bv = v; bi = e; }
      }
    }
  }
  block_best(bv, bi, sv, si);
  if (threadIdx.x == 0) cand[r * kArgmaxSlices + j] = make_float2(bv, __int_as_float(bi));
}

__global__ void argmax_merge_kernel(const float2* __restrict__ cand, int n_slices, int rows, int* __restrict__ amax) {
  pdl_wait();
  pdl_launch_dependents();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= rows) return;
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  for (int j = 0; j < n_slices; ++j) {
    const float2 e = cand[r * kArgmaxSlices + j];
    const int id = __float_as_int(e.y);
    if (better(e.x, id, bv, bi)) { bv = e.x; bi = id; }
  }
  amax[r] = bi;
}

void launch_argmax_rows(PartialView P, int vocab, int rows, int* amax, float* logits_out, float* cand, cudaStream_t st) {
  const int vec = vocab % 4 == 0 && P.ld % 4 == 0;
  int chunk = (vocab + kArgmaxSlices - 1) / kArgmaxSlices;
  chunk = (chunk + 3) / 4 * 4;
  const int n_slices = (vocab + chunk - 1) / chunk;
  launch_pdl(argmax_slice_kernel, dim3(rows, n_slices), dim3(256), 0, st, P, vocab, chunk, reinterpret_cast<float2*>(cand), logits_out, vec);
  launch_pdl(argmax_merge_kernel, dim3((rows + 127) / 128), dim3(128), 0, st, reinterpret_cast<const float2*>(cand), n_slices, rows, amax);
}

// --------------------------------------------------------------------------------------------
// control: tree tokens, acceptance, compaction
// --------------------------------------------------------------------------------------------
// The tree of every sequence laid out again with the caller's tokens (entries < 0 keep the drafted ones).
__global__ void tree_override_kernel(const TopkTreeArgs a, const int* __restrict__ override_tok) {
  pdl_wait();
  pdl_launch_dependents();
  const int b = blockIdx.x;
  tree_row(a.tree, reinterpret_cast<const DevState*>(a.state + a.state_stride * b), nullptr, override_tok + (size_t)b * a.rows,
           a.tok + (size_t)b * a.rows, reinterpret_cast<RowMeta*>(a.meta + a.meta_stride * b), threadIdx.x);
}

void launch_tree_override(const TopkTreeArgs& a, const int* override_tok, int batch, cudaStream_t st) {
  launch_pdl(tree_override_kernel, dim3(batch), dim3(kMaxRows), 0, st, a, override_tok);
}

// Greedy acceptance: node n matches if its token equals the target's choice at its parent; it is
// accepted if every node on its root path matches; the deepest accepted node wins (lowest index
// among equals).  The match set is a 128-bit mask tested against the ancestor masks.
// Compaction: slot C + j <- slot C + path[j] in every layer's cache, accepted hidden rows to the next draft's queue.
//
// One launch for all sequences (blockIdx.y).  Every block finds the accepted path for itself (tokens, choices and tree are a
// few KB of L2; C is the row table's base, since one block moves the state on), then moves its own piece: one block per layer
// and K / V half, one per queued hidden row.  Bound: latency (two dependent L2 round trips and the copy's own).
// 16-byte copies with all of a thread's loads issued before its first store.  A launch for the acceptance and, per sequence,
// one of a block per layer that copied 2-byte elements in path order cost a step 12 us more at 7B (31 us of them on the
// chain, part of them hidden behind the next graph launch) and 345 us more with eight sequences.
template <typename T>
__global__ void __launch_bounds__(256)
accept_compact_kernel(const AcceptArgs a) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ u64 match[2];
  __shared__ int best_key, L_s;
  __shared__ int path_s[kPendMax];
  const TreeDev* tree = a.tree;
  const int b = blockIdx.y, n = threadIdx.x, N = tree->n_nodes;
  const int* tok = a.tok + (size_t)b * a.rows;
  const int* amax = a.amax + (size_t)b * a.rows;
  const int C = reinterpret_cast<const RowMeta*>(a.meta + a.meta_stride * b)->base;
  if (n < 2) match[n] = 0ull;
  if (n == 0) best_key = 0;
  u64 anc0 = 0, anc1 = 0;
  bool m = false;
  if (n < N) {
    anc0 = tree->anc[n][0];
    anc1 = tree->anc[n][1];
    m = n == 0 || tok[n] == amax[tree->parent[n]];
  }
  __syncthreads();
  const unsigned votes = __ballot_sync(0xffffffffu, m);
  if ((n & 31) == 0 && n < kMaxRows) atomicOr(&match[n >> 6], (u64)votes << (n & 32));
  __syncthreads();
  if (n < N && ((anc0 & ~match[0]) | (anc1 & ~match[1])) == 0ull) atomicMax(&best_key, tree->depth[n] * 256 + (255 - n));
  __syncthreads();
  const int best = 255 - (best_key & 255);
  if (n == best) {                                     // the ancestors of the deepest accepted node, in node order
    int L = 0;
    while (anc0 && L < kPendMax) { path_s[L++] = __ffsll((long long)anc0) - 1; anc0 &= anc0 - 1; }
    while (anc1 && L < kPendMax) { path_s[L++] = 64 + __ffsll((long long)anc1) - 1; anc1 &= anc1 - 1; }
    L_s = L;
  }
  __syncthreads();
  const int L = L_s;
  if ((int)blockIdx.x < 2 * a.n_layers) {
    // path is strictly increasing with path[j] >= j, so no source slot is the destination of an earlier move
    const KvView kv = reinterpret_cast<const KvView*>(a.kv_tab + a.kv_tab_stride * b)[blockIdx.x >> 1];
    T* cache = (T*)((blockIdx.x & 1) ? kv.v : kv.k);
    constexpr int E = 16 / sizeof(T);
    const int per_head = a.dh / E, items = a.n_heads * per_head;
    for (int i = n; i < items; i += blockDim.x) {
      const int h = i / per_head;
      uint4* base = reinterpret_cast<uint4*>(cache + ((size_t)h * a.max_ctx + C) * a.dh + (i - h * per_head) * E);
      uint4 v[kPendMax];
#pragma unroll
      for (int j = 1; j < kPendMax; ++j)
        if (j < L && path_s[j] != j && C + path_s[j] < a.max_ctx) v[j] = base[(size_t)path_s[j] * per_head];
#pragma unroll
      for (int j = 1; j < kPendMax; ++j)
        if (j < L && path_s[j] != j && C + path_s[j] < a.max_ctx) base[(size_t)j * per_head] = v[j];
    }
    return;
  }
  const int j = blockIdx.x - 2 * a.n_layers;           // queued hidden row
  if (j < L) {
    const float* src = a.hidden + ((size_t)b * a.rows + path_s[j]) * a.d;
    float* dst = a.pend_h + ((size_t)b * a.pend_rows + j) * a.d;
    for (int c = n * 4; c < a.d; c += blockDim.x * 4) store4(dst + c, load4(src + c));
  }
  if (j == 0 && n == 0) {
    DevState* s = reinterpret_cast<DevState*>(a.state + a.state_stride * b);
    const int nr = amax[best];
    for (int i = 0; i < kPendMax; ++i) {
      s->path[i] = i < L ? path_s[i] : -1;
      s->out_tok[i] = i < L ? tok[path_s[i]] : -1;
      if (i < L) s->pend_tok[i] = i + 1 < L ? tok[path_s[i + 1]] : nr;
    }
    s->L = L;
    s->C_old = C;
    s->best = best;
    s->next_root = nr;
    s->C = C + L;
    s->root = nr;
    s->n_pending = L;
    s->step += 1;
    for (int i = 0; a.out_tokens != nullptr && i < a.out_k; ++i) a.out_tokens[b * a.out_k + i] = i < L ? tok[path_s[i]] : -1;
    if (a.out_n != nullptr) a.out_n[b] = L;
  }
}

const void* accept_compact_function(int dtype) {
  return dtype == AMPH_DTYPE_F32 ? (const void*)accept_compact_kernel<float> : (const void*)accept_compact_kernel<bf16>;
}

void launch_accept_compact(const AcceptArgs& a, int batch, int dtype, cudaStream_t st) {
  AMPH_DISPATCH(dtype, launch_pdl(accept_compact_kernel<T>, dim3(2 * a.n_layers + kPendMax, batch), dim3(256), 0, st, a));
}

// --------------------------------------------------------------------------------------------
// Sampling at a temperature (Table 2; Section 2, rejection sampling with point-mass proposals)
// --------------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al., SC'11): ten rounds; each multiplies counter words 0 and 2 by fixed odd constants,
// crosses the halves of the 64-bit products and mixes in the key, which is bumped by Weyl constants between rounds.
__device__ __forceinline__ uint32_t philox_first_word(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
    const uint32_t h0 = __umulhi(0xD2511F53u, c0), l0 = 0xD2511F53u * c0;
    const uint32_t h1 = __umulhi(0xCD9E8D57u, c2), l1 = 0xCD9E8D57u * c2;
    const uint32_t n0 = h1 ^ c1 ^ k0, n2 = h0 ^ c3 ^ k1;
    c0 = n0; c1 = l1; c2 = n2; c3 = l0;
  }
  return c0;
}

constexpr int kSampleThreads = 1024;
constexpr int kSampleWarps = kSampleThreads / 32;
constexpr int kSampleMaxChildren = 16;       // candidates a head keeps at most = children a node has at most

// One block per row and sequence (blockIdx.y).  w(v) = exp((l_v - max) / T); the row's uniform scaled by the sum of all weights
// is compared with running sums of w, so nothing is divided.  Every thread owns a contiguous range of ids; sums over threads
// are block-wide scans in a fixed order (deterministic).  Bound: latency, then the logits' L2 reads: with the children
// collected and the range sums added one after the other by one thread, and a launch per sequence, a step of eight sequences
// of 48 rows took 410 us more (32000 ids).
__global__ void __launch_bounds__(kSampleThreads)
sample_rows_kernel(const float* __restrict__ logits, int vocab, int row0, int rows_per, const TreeDev* __restrict__ tree,
                   const int* __restrict__ tok, const char* __restrict__ state, size_t state_stride, int seq0, int stream_id, float inv_t,
                   uint32_t k0, uint32_t k1, int* __restrict__ choice, float* __restrict__ uniforms_out) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ float red[kSampleWarps];
  __shared__ int kids_all[kMaxRows];
  __shared__ int kid_tok[kSampleMaxChildren];
  __shared__ float kid_w[kSampleMaxChildren];
  __shared__ uint32_t kid_votes[kMaxRows / 32];
  __shared__ int n_kids_s, result_s, owner_s, last_s;
  __shared__ float target_s, base_s;
  const int r = blockIdx.x, b = blockIdx.y, row = row0 + b * rows_per + r, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const float* l = logits + (size_t)row * vocab;
  const bool vec = vocab % 4 == 0;
  // row maximum; meanwhile the first warps find the row's children
  float m = -INFINITY;
  if (vec) {
    for (int v = tid * 4; v < vocab; v += kSampleThreads * 4) {
      const float4 x = load4(l + v);
      m = fmaxf(m, fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)));
    }
  } else {
    for (int v = tid; v < vocab; v += kSampleThreads) m = fmaxf(m, l[v]);
  }
  const bool kids_given = tree != nullptr && tok != nullptr;
  bool is_kid = false;
  if (tid < kMaxRows) {
    is_kid = kids_given && tid > r && tid < tree->n_nodes && tree->parent[tid] == r;
    const uint32_t v = __ballot_sync(0xffffffffu, is_kid);
    if (lane == 0) kid_votes[warp] = v;
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) red[warp] = m;
  if (tid == 0) { result_s = -1; owner_s = kSampleThreads; last_s = -1; }
  __syncthreads();
  m = red[lane];
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (is_kid) {                                            // node order = order of the votes
    int at = __popc(kid_votes[warp] & ((1u << lane) - 1u));
    for (int w = 0; w < warp; ++w) at += __popc(kid_votes[w]);
    kids_all[at] = tok[(size_t)b * rows_per + tid];
  }
  __syncthreads();
  if (tid == 0) {                                          // the distinct tokens of the row's children, in node order
    int n = 0, nk = 0;
    for (int w = 0; w < kMaxRows / 32; ++w) n += __popc(kid_votes[w]);
    for (int c = 0; c < n && nk < kSampleMaxChildren; ++c) {
      const int x = kids_all[c];
      bool seen = x < 0 || x >= vocab;
      for (int j = 0; j < nk; ++j) seen = seen || kid_tok[j] == x;
      if (!seen) kid_tok[nk++] = x;
    }
    n_kids_s = nk;
  }
  __syncthreads();
  const int nk = n_kids_s;
  if (tid < nk) kid_w[tid] = __expf((l[kid_tok[tid]] - m) * inv_t);
  // this thread's ids (whole groups of four); its weight sum leaves the children's tokens out
  const int chunk = ((vocab + kSampleThreads - 1) / kSampleThreads + 3) / 4 * 4;
  const int lo = tid * chunk, hi = lo + chunk < vocab ? lo + chunk : vocab;
  bool kid_here = false;
  for (int j = 0; j < nk; ++j) kid_here = kid_here || (kid_tok[j] >= lo && kid_tok[j] < hi);
  float mine = 0.f;
  if (kid_here || !vec) {
    for (int v = lo; v < hi; ++v) {
      bool kid = false;
      for (int j = 0; j < nk; ++j) kid = kid || kid_tok[j] == v;
      if (!kid) mine += __expf((l[v] - m) * inv_t);
    }
  } else {
    for (int v = lo; v < hi; v += 4) {                     // vocab % 4 == 0: the last group is whole
      const float4 x = load4(l + v);
      mine += __expf((x.x - m) * inv_t);
      mine += __expf((x.y - m) * inv_t);
      mine += __expf((x.z - m) * inv_t);
      mine += __expf((x.w - m) * inv_t);
    }
  }
  // inclusive scan of the range sums over the block
  float run = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const float up = __shfl_up_sync(0xffffffffu, run, o);
    if (lane >= o) run += up;
  }
  if (lane == 31) red[warp] = run;                         // every thread has read the maxima before the two barriers above
  __syncthreads();
  float wsum = red[lane];
  for (int o = 1; o < 32; o <<= 1) {
    const float up = __shfl_up_sync(0xffffffffu, wsum, o);
    if (lane >= o) wsum += up;
  }
  const float rest = __shfl_sync(0xffffffffu, wsum, 31);
  const float below = __shfl_sync(0xffffffffu, wsum, warp == 0 ? 0 : warp - 1);
  const float before = warp == 0 ? 0.f : below;
  if (tid == 0) {
    const DevState* s = reinterpret_cast<const DevState*>(state + state_stride * b);
    const uint32_t w = philox_first_word((uint32_t)r, (uint32_t)s->step, (uint32_t)(seq0 + b), (uint32_t)stream_id, k0, k1);
    const float u = (float)(w >> 8) * (1.0f / 16777216.0f);
    if (uniforms_out) uniforms_out[b * rows_per + r] = u;
    float kids = 0.f;
    for (int j = 0; j < nk; ++j) kids += kid_w[j];
    const float target = u * (kids + rest);
    float acc = 0.f;
    int res = -1;
    for (int j = 0; j < nk && res < 0; ++j) {            // children first: accepted iff the running sum passes the target
      acc += kid_w[j];
      if (target < acc) res = kid_tok[j];
    }
    result_s = res;
    target_s = target;
    base_s = kids;
  }
  __syncthreads();
  if (result_s >= 0) {
    if (tid == 0) choice[row] = result_s;
    return;
  }
  // residual distribution: the first id, ascending, children's tokens left out, whose running sum exceeds the target
  if (mine > 0.f) {
    if (base_s + (before + run) > target_s) atomicMin(&owner_s, tid);
    atomicMax(&last_s, tid);
  }
  __syncthreads();
  const bool beyond = owner_s == kSampleThreads;           // rounding left the target above the total: the last admissible id
  if (tid == (beyond ? last_s : owner_s)) {
    float acc = beyond ? -INFINITY : base_s + (before + (run - mine));
    int res = -1, last = -1;
    for (int v = lo; v < hi; ++v) {
      bool kid = false;
      for (int j = 0; j < nk; ++j) kid = kid || kid_tok[j] == v;
      if (kid) continue;
      const float w = __expf((l[v] - m) * inv_t);
      if (w > 0.f) last = v;
      acc += w;
      if (acc > target_s) { res = v; break; }
    }
    choice[row] = res >= 0 ? res : last;
  }
}

void launch_sample_rows(const float* logits, int vocab, int row0, int n_rows, int rows_per, int batch, const TreeDev* tree, const int* tok,
                        const void* state, size_t state_stride, int seq0, int stream_id, float temperature, unsigned long long seed,
                        int* choice, float* uniforms_out, cudaStream_t st) {
  launch_pdl(sample_rows_kernel, dim3(n_rows, batch), dim3(kSampleThreads), 0, st, logits, vocab, row0, rows_per, tree, tok,
             (const char*)state, state_stride, seq0, stream_id, 1.0f / temperature, (uint32_t)(seed & 0xffffffffull), (uint32_t)(seed >> 32),
             choice, uniforms_out);
}

// Grid (512-column chunk, row).  Bound: L2 (the splits' sums were just written); the loads of all splits are in flight together.
__global__ void __launch_bounds__(128)
reduce_partials_kernel(PartialView P, float* __restrict__ y, int cols, int vec, int* err, int* status) {
  pdl_wait();
  pdl_launch_dependents();
  if (err != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
    if (status != nullptr) *status = *err;
    *err = 0;
  }
  const int r = blockIdx.y, c = (blockIdx.x * 128 + threadIdx.x) * 4;
  if (vec) {
    if (c < cols) store4(y + (size_t)r * cols + c, sum_partials4_wide(P, r, c));
  } else {
    for (int e = c; e < cols && e < c + 4; ++e) y[(size_t)r * cols + e] = sum_partials(P, r, e);
  }
}

void launch_reduce_partials(PartialView P, float* y, int rows, int cols, cudaStream_t st, int* err, int* status) {
  const int vec = cols % 4 == 0 && P.ld % 4 == 0 && P.split_stride % 4 == 0 && ((uintptr_t)y & 15) == 0;
  launch_pdl(reduce_partials_kernel, dim3((cols + 511) / 512, rows), dim3(128), 0, st, P, y, cols, vec, err, status);
}

template <typename T>
__global__ void kv_export_kernel(const T* __restrict__ c, int row0, int n_heads, int dh, int max_ctx,
                                 float* __restrict__ dst) {
  pdl_wait();
  pdl_launch_dependents();
  const int slot = row0 + blockIdx.x;
  for (int i = threadIdx.x; i < n_heads * dh; i += blockDim.x) {
    const int h = i / dh, e = i - h * dh;
    dst[(size_t)blockIdx.x * n_heads * dh + i] = to_f(c[((size_t)h * max_ctx + slot) * dh + e]);
  }
}

void launch_kv_export(KvView kv, int which, int dtype, int row0, int rows, int n_heads, int head_dim, int max_ctx,
                      float* dst, cudaStream_t st) {
  if (rows <= 0) return;
  AMPH_DISPATCH(dtype, launch_pdl(kv_export_kernel<T>, dim3(rows), dim3(256), 0, st, (const T*)(which ? kv.v : kv.k), row0, n_heads,
                                                                 head_dim, max_ctx, dst));
}

// End of prefill: root = greedy choice after the last prompt token; the last prompt row stays
// pending so that the first draft runs the adaptation layers on it (Eq. 1).
__global__ void prefill_tail_kernel(DevState* s, const int* __restrict__ amax, int last_row,
                                    const float* __restrict__ hidden, float* __restrict__ pend_h, int d, int C) {
  pdl_wait();
  pdl_launch_dependents();
  for (int c = threadIdx.x; c < d; c += blockDim.x) pend_h[c] = hidden[(size_t)last_row * d + c];
  if (threadIdx.x == 0) {
    const int root = amax[last_row];
    s->C = C;
    s->root = root;
    s->n_pending = 1;
    s->pend_tok[0] = root;
    s->L = 0;
    s->C_old = C;
    s->best = 0;
    s->next_root = root;
    s->step = 0;
  }
}

void launch_prefill_tail(DevState* s, const int* amax, int last_row, const float* hidden, float* pend_h, int d,
                         int C, cudaStream_t st) {
  launch_pdl(prefill_tail_kernel, dim3(1), dim3(256), 0, st, s, amax, last_row, hidden, pend_h, d, C);
}

}  // namespace amph
