// bf16 projections of up to 64 activation rows (gate / up: 128) whose epilogue needs the whole sum:  Y[rows][out] = X . W^T.
//
// The activation rows are the MMA operand A (M = 64, or 128), the weight rows operand B (N = 8 .. 256 of them, a multiple of 8), so a
// tile may have any height that spreads a matrix evenly over the SMs, and a thread of the epilogue holds neighbouring features
// of a row: gate and up of a feature, or both members of a rotation pair, meet in one thread's registers.  A CTA owns the whole
// K range of its tile.  Weights and activations have a ring each: weights come from HBM and need many bytes in flight,
// activations come from L2 and need few.
//
// Ring positions and parities are counted, and the stages' MMAs unrolled: two divisions by run-time values in the loop that issues
// them are 350 clocks, as much as ten MMAs of this size; a gate / up launch of 180 MB took 40.7 us with them, 30.9 without.
//
// Warp roles: 0 = TMA producer of the weights (waits for no other kernel), 1 = MMA issuer (owns the tensor memory), 2-5 =
// epilogue, 6 = TMA producer of the activations.  Every barrier wait is bounded, counted from the end of the kernel ahead: if one gives
// up the CTA raises the error flag, lets its copies land and its MMAs finish and leaves; its outputs are finite then (sums of zero).
#include "gemm_tc_common.cuh"

namespace amph {

using namespace tc;

namespace {

constexpr int kRowsThreads = 224;
constexpr int kMaxRing = 12;

enum { ROWS_SWIGLU = 0, ROWS_ROPE = 1, ROWS_RESID = 2 };

struct RowsMaps {
  CUtensorMap w[3];
  CUtensorMap x;
};

struct RowsParams {
  int tiles_per_seg;        // tiles of one matrix (ROPE: of q, k, v each)
  int kblocks;
  int half;                 // weight rows of one half of a tile (SWIGLU: gate or up; ROPE: one half of the pairs); RESID: the tile
  int n;                    // weight rows of a tile: N of the MMA
  int nt;                   // rows of an activation box (a multiple of 16, at most M)
  int kb_cut;               // M = 128: K blocks from here on go to an accumulator of their own (kblocks: there is one only)
  int rows;
  int w_stages, x_stages;
  int l2_prefetch;          // weight stages beyond the ring that are asked into L2 ahead of the dependency
  int tmem_cols;
  RowScale rs;
  __nv_bfloat16* act;       // SWIGLU: [rows][f]
  int f;
  int up_first;             // the tensor map's outer index 0 is the up matrix
  __nv_bfloat16* q;         // ROPE: [rows][n_heads * dh]
  __nv_bfloat16* kc;        // [n_heads][max_ctx][dh]
  __nv_bfloat16* vc;
  const RowMeta* meta;
  const float2* rope;       // [rows][dh / 2] (cos, sin)
  int n_heads, dh, max_ctx;
  float* x;                 // RESID: [rows][out], updated in place
  const __nv_bfloat16* gain;      // or NULL: x only
  __nv_bfloat16* xn;
  float* ss;                // [row][tiles] sums of squares
  int out;
  int* err_flag;
  unsigned long long wait_limit_ns;
  uint32_t extra_tx;        // self-test only: bytes the first stage's barrier expects beyond what is copied
};

__device__ __forceinline__ void load_w(void* dst, const CUtensorMap* map, int row, int kb, uint64_t* bar, uint64_t pol, bool pair) {
  if (pair)                                          // (column, row, matrix or half, K block)
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
        ::"r"(smem_u32(dst)), "l"(map), "r"(0), "r"(row), "r"(0), "r"(kb), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;"
        ::"r"(smem_u32(dst)), "l"(map), "r"(0), "r"(row), "r"(kb), "r"(smem_u32(bar)), "l"(pol)
        : "memory");
}
__device__ __forceinline__ void prefetch_w(const CUtensorMap* map, int row, int kb, bool pair) {
  if (pair) asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];" ::"l"(map), "r"(0), "r"(row), "r"(0), "r"(kb) : "memory");
  else asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(map), "r"(0), "r"(row), "r"(kb) : "memory");
}
__device__ __forceinline__ void load_x(void* dst, const CUtensorMap* map, int kb, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(0), "r"(0), "r"(kb), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// 16 TMEM lanes x 8 columns over the whole warp: thread t, value 2 * hi + e holds lane t / 4 + 8 * hi, column 2 * (t % 4) + e
// (an MMA accumulator fragment).
__device__ __forceinline__ void ld_frag8(uint32_t taddr, float* v) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(taddr) : "memory");
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

template <int EPI, int KS, int M>
__global__ void __launch_bounds__(kRowsThreads)
tc_rows_kernel(const __grid_constant__ RowsMaps maps, const RowsParams prm) {
  constexpr bool PAIR = EPI != ROWS_RESID;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  static_assert(M == 64 || (KS == 1 && EPI == ROWS_SWIGLU), "a cut between two accumulators falls between two stages");
  __shared__ float inv_s[PAIR ? M : 1];                            // 1 / rms of the activation rows
  __shared__ __align__(8) uint64_t w_full[kMaxRing], w_empty[kMaxRing], x_full[kMaxRing], x_empty[kMaxRing], accum_bar, drain_bar;
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;

  const unsigned long long limit_ns = prm.wait_limit_ns;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tile = blockIdx.x, seg = tile / prm.tiles_per_seg, lt = tile - seg * prm.tiles_per_seg;
  int row0 = lt * prm.half;                                        // first weight row (of the lower half) in its matrix
  if constexpr (EPI == ROWS_ROPE) {
    const int tph = (prm.dh >> 1) / prm.half;                      // tiles per head
    row0 = lt / tph * prm.dh + lt % tph * prm.half;
  }
  const int its = (prm.kblocks + KS - 1) / KS;
  const uint32_t w_tile = (uint32_t)prm.n * 128, x_tile = (uint32_t)prm.nt * 128;       // one K block of each operand
  const uint32_t w_bytes = w_tile * KS, x_bytes = x_tile * KS;
  uint8_t* const xs = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* const ws = xs + (size_t)prm.x_stages * x_bytes;         // behind the activations: an MMA reads M rows whatever nt is

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < prm.w_stages; ++s) { mbar_init(&w_full[s], 1); mbar_init(&w_empty[s], 1); }
    for (int s = 0; s < prm.x_stages; ++s) { mbar_init(&x_full[s], 1); mbar_init(&x_empty[s], 1); }
    mbar_init(&accum_bar, 1);
    mbar_init(&drain_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // Barrier 2 tells the warps that use the mbarriers that they exist, barrier 3 the epilogue that the accumulator does.
  if (warp == 0) { __syncwarp(); asm volatile("bar.arrive 2, 96;" ::: "memory"); }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(prm.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    pdl_launch_dependents();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncwarp();
  if (warp < 2) asm volatile("bar.arrive 3, 192;" ::: "memory");
  else if (warp < 6) asm volatile("bar.sync 3, 192;" ::: "memory");
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");

  if (warp == 0) {
    // ---------------- weights: they depend on nothing, so the ring fills while the kernel before this one still runs
    const bool leader = elect_one();
    const uint64_t pol = l2_evict_first_policy();
    const CUtensorMap* map = &maps.w[seg];
    if (leader) asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
    int issued = 0;
    for (int i = 0, s = 0, ph = 1; i < its; ++i) {
      if (i == prm.w_stages) pdl_wait();             // the time spent behind the kernel ahead does not count for the limit
      if (i >= prm.w_stages && !__all_sync(0xffffffffu, mbar_wait(&w_empty[s], ph, &abort_flag, limit_ns))) break;
      if (leader) {
        mbar_expect_tx(&w_full[s], w_bytes + (i == 0 ? prm.extra_tx : 0u));
        load_w(ws + (size_t)s * w_bytes, map, row0, i * KS, &w_full[s], pol, PAIR);
        if (i == prm.w_stages - 1)
          for (int j = 1; j <= prm.l2_prefetch && i + j < its; ++j) prefetch_w(map, row0, (i + j) * KS, PAIR);
      }
      __syncwarp();
      issued = i + 1;
      if (++s == prm.w_stages) { s = 0; ph ^= 1; }
    }
    if (abort_flag && lane == 0)                       // let every copy that was issued land
      for (int i = issued > prm.w_stages ? issued - prm.w_stages : 0; i < issued; ++i) {
        const unsigned long long t0 = now_ns();
        while (!mbar_try(&w_full[i % prm.w_stages], (i / prm.w_stages) & 1) && now_ns() - t0 < kDrainNs) {}
      }
  } else if (warp == 6) {
    // ---------------- activations
    const bool leader = elect_one();
    if (leader) asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.x) : "memory");
    pdl_wait();
    asm volatile("bar.sync 2, 96;" ::: "memory");
    int issued = 0;
    for (int i = 0, s = 0, ph = 1; i < its; ++i) {
      if (i >= prm.x_stages && !__all_sync(0xffffffffu, mbar_wait(&x_empty[s], ph, &abort_flag, limit_ns))) break;
      if (leader) {
        mbar_expect_tx(&x_full[s], x_bytes);
        load_x(xs + (size_t)s * x_bytes, &maps.x, i * KS, &x_full[s]);
      }
      __syncwarp();
      issued = i + 1;
      if (++s == prm.x_stages) { s = 0; ph ^= 1; }
    }
    if (abort_flag && lane == 0)
      for (int i = issued > prm.x_stages ? issued - prm.x_stages : 0; i < issued; ++i) {
        const unsigned long long t0 = now_ns();
        while (!mbar_try(&x_full[i % prm.x_stages], (i / prm.x_stages) & 1) && now_ns() - t0 < kDrainNs) {}
      }
  } else if (warp == 1) {
    // ---------------- MMA issuer (the warp stays converged, its elected lane issues)
    const bool leader = elect_one();
    pdl_wait();
    asm volatile("bar.sync 2, 96;" ::: "memory");
    const uint32_t tmem_d = tmem_base_slot;
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(prm.n >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
    const uint32_t xa = smem_u32(xs), wa = smem_u32(ws);
    const uint64_t ad0 = umma_desc(xa), bd0 = umma_desc(wa);       // the address is the descriptor's lowest field, in 16 bytes
    bool ok = true;
    int wst = 0, wph = 0, xst = 0, xph = 0;
    for (int i = 0; i < its; ++i) {
      ok = __all_sync(0xffffffffu, mbar_wait(&w_full[wst], wph, &abort_flag, limit_ns) && mbar_wait(&x_full[xst], xph, &abort_flag, limit_ns));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (leader) {
        uint64_t ad = ad0 + (uint64_t)((uint32_t)xst * x_bytes >> 4), bd = bd0 + (uint64_t)((uint32_t)wst * w_bytes >> 4);
#pragma unroll
        for (int kk = 0; kk < KS; ++kk, ad += x_tile >> 4, bd += w_tile >> 4) {      // K blocks past the end are zeros
#pragma unroll
          for (int k = 0; k < kTileK / kUmmaK; ++k) {
            if constexpr (M == 64) mma(tmem_d, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), idesc, (i | kk | k) ? 1u : 0u);
            else mma(tmem_d + (i >= prm.kb_cut ? (uint32_t)prm.n : 0u), ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), idesc, (i != 0 && i != prm.kb_cut) || k ? 1u : 0u);
          }
        }
        commit(&w_empty[wst]);
        commit(&x_empty[xst]);
      }
      __syncwarp();
      if (++wst == prm.w_stages) { wst = 0; wph ^= 1; }
      if (++xst == prm.x_stages) { xst = 0; xph ^= 1; }
    }
    if (ok && leader) commit(&accum_bar);
    if (!ok) {                                       // no tensor memory is given back under an MMA
      if (leader) commit(&drain_bar);
      __syncwarp();
      const unsigned long long t0 = now_ns();
      while (!mbar_try(&drain_bar, 0) && now_ns() - t0 < kDrainNs) {}
    }
    __syncwarp();
  } else {
    // ---------------- epilogue: row r of the accumulator sits in TMEM lane 32 (r / 16) + r % 16 (M = 64), or r (M = 128); the warp of
    // quarter q takes 16 rows at a time, this thread ra and rb of them, columns 8 j + 2 (lane % 4) and the next one
    const int quarter = warp & 3, cq = 2 * (lane & 3);
    pdl_wait();
    if constexpr (PAIR) {
      const int et = threadIdx.x - 64;
      if (et < prm.rows) inv_s[et] = row_scale(prm.rs, et);
      asm volatile("bar.sync 1, 128;" ::: "memory");
    }
    constexpr int U = 4;                               // pieces of 8 columns in flight
    auto sums_ready = [&] {
      const bool ok = __all_sync(0xffffffffu, mbar_wait(&accum_bar, 0, &abort_flag, limit_ns));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      return ok;
    };
    const bool two = M == 128 && prm.kb_cut < prm.kblocks;
    for (int part = 0; part < M / 64; ++part) {
      const int ra = quarter * (M / 4) + part * 16 + (lane >> 2), rb = ra + 8;
      const bool la = ra < prm.rows, lb = rb < prm.rows;
      const uint32_t taddr = tmem_base_slot + ((uint32_t)(quarter * 32 + part * 16) << 16);
      // the second accumulator's sums join the first one's, in the order in which split-K sums are added
      auto join = [&](uint32_t at, float (*v)[4], int c0) {
        if constexpr (M == 128) {
          if (!two) return;
          float w[U][4];
#pragma unroll
          for (int j = 0; j < U; ++j)
            if (c0 + 8 * j < prm.half) ld_frag8(at + (uint32_t)prm.n + c0 + 8 * j, w[j]);
          ld_wait();
#pragma unroll
          for (int j = 0; j < U; ++j)
            if (c0 + 8 * j < prm.half) { v[j][0] += w[j][0]; v[j][1] += w[j][1]; v[j][2] += w[j][2]; v[j][3] += w[j][3]; }
        }
      };
      if constexpr (EPI == ROWS_SWIGLU) {
        const float sa = la ? inv_s[ra] : 0.f, sb = lb ? inv_s[rb] : 0.f;
        const bool ok = sums_ready();
        const uint32_t tg = taddr + (prm.up_first ? (uint32_t)prm.half : 0u), tu = taddr + (prm.up_first ? 0u : (uint32_t)prm.half);
        __nv_bfloat16* const pa = prm.act + (size_t)ra * prm.f + row0 + cq;
        __nv_bfloat16* const pb = prm.act + (size_t)rb * prm.f + row0 + cq;
        // M = 128 stands for split-K sums and swiglu_kernel, whose exponential and division it keeps
        auto glu = [](float g, float u, float sc) {
          const float t = g * sc;
          if constexpr (M == 128) return t / (1.0f + expf(-t)) * (u * sc);
          else return __fdividef(t, 1.0f + __expf(-t)) * (u * sc);
        };
        for (int c0 = 0; c0 < prm.half; c0 += 8 * U) {
          float g[U][4], u[U][4];
#pragma unroll
          for (int j = 0; j < U; ++j)
            if (c0 + 8 * j < prm.half) { ld_frag8(tg + c0 + 8 * j, g[j]); ld_frag8(tu + c0 + 8 * j, u[j]); }
          ld_wait();
          join(tg, g, c0);
          join(tu, u, c0);
#pragma unroll
          for (int j = 0; j < U; ++j) {
            const int c = c0 + 8 * j;
            if (c < prm.half && row0 + c < prm.f) {
              const uint32_t ya = ok ? pack2(glu(g[j][0], u[j][0], sa), glu(g[j][1], u[j][1], sa)) : 0u;
              const uint32_t yb = ok ? pack2(glu(g[j][2], u[j][2], sb), glu(g[j][3], u[j][3], sb)) : 0u;
              if (la) *reinterpret_cast<uint32_t*>(pa + c) = ya;
              if (lb) *reinterpret_cast<uint32_t*>(pb + c) = yb;
            }
          }
        }
      } else if constexpr (EPI == ROWS_ROPE) {
        const float sa = la ? inv_s[ra] : 0.f, sb = lb ? inv_s[rb] : 0.f;
        const int hdim = prm.dh >> 1, h = row0 / prm.dh, i0 = row0 - h * prm.dh + cq;      // head, this thread's first pair
        __nv_bfloat16 *da = nullptr, *db = nullptr;
        if (seg == 0) {
          da = prm.q + (size_t)ra * prm.n_heads * prm.dh + h * prm.dh + i0;
          db = prm.q + (size_t)rb * prm.n_heads * prm.dh + h * prm.dh + i0;
          if (!la) da = nullptr;
          if (!lb) db = nullptr;
        } else {
          __nv_bfloat16* const cache = (seg == 1 ? prm.kc : prm.vc) + (size_t)h * prm.max_ctx * prm.dh + i0;
          const int n_rows = prm.meta->n_rows;
          const int pa = la && ra < n_rows ? prm.meta->slot[ra] : -1, pb = lb && rb < n_rows ? prm.meta->slot[rb] : -1;
          if (pa >= 0 && pa < prm.max_ctx) da = cache + (size_t)pa * prm.dh;
          if (pb >= 0 && pb < prm.max_ctx) db = cache + (size_t)pb * prm.dh;
        }
        const float2* const ta = prm.rope + (size_t)ra * hdim + i0;
        const float2* const tb = prm.rope + (size_t)rb * hdim + i0;
        const float4 unit = make_float4(1.f, 0.f, 1.f, 0.f);
        const bool ok = sums_ready();
        for (int c0 = 0; c0 < prm.half; c0 += 8 * U) {
          float lo[U][4], hi[U][4];
          float4 ca[U], cb[U];
#pragma unroll
          for (int j = 0; j < U; ++j) {
            const int c = c0 + 8 * j;
            if (c < prm.half) { ld_frag8(taddr + c, lo[j]); ld_frag8(taddr + prm.half + c, hi[j]); }
            ca[j] = seg < 2 && la && c < prm.half ? *reinterpret_cast<const float4*>(ta + c) : unit;       // (cos, sin) of two pairs
            cb[j] = seg < 2 && lb && c < prm.half ? *reinterpret_cast<const float4*>(tb + c) : unit;
          }
          ld_wait();
#pragma unroll
          for (int j = 0; j < U; ++j) {
            const int c = c0 + 8 * j;
            if (c >= prm.half) continue;
            auto put = [&](__nv_bfloat16* dst, float a0, float a1, float b0, float b1, const float4& cs, float sc) {
              if (dst == nullptr) return;
              if (!ok) { a0 = a1 = b0 = b1 = 0.f; }
              a0 *= sc; a1 *= sc; b0 *= sc; b1 *= sc;
              const uint32_t l = seg < 2 ? pack2(a0 * cs.x - b0 * cs.y, a1 * cs.z - b1 * cs.w) : pack2(a0, a1);
              const uint32_t u = seg < 2 ? pack2(b0 * cs.x + a0 * cs.y, b1 * cs.z + a1 * cs.w) : pack2(b0, b1);
              *reinterpret_cast<uint32_t*>(dst + c) = l;
              *reinterpret_cast<uint32_t*>(dst + hdim + c) = u;
            };
            put(da, lo[j][0], lo[j][1], hi[j][0], hi[j][1], ca[j], sa);
            put(db, lo[j][2], lo[j][3], hi[j][2], hi[j][3], cb[j], sb);
          }
        }
      } else {
        // residual update; the tile has at most 8 U features, their old values are fetched under the main loop
        const int f0 = row0 + cq;
        float* const xa = prm.x + (size_t)ra * prm.out + f0;
        float* const xb = prm.x + (size_t)rb * prm.out + f0;
        float2 oa[U], ob[U], gn[U];
#pragma unroll
        for (int j = 0; j < U; ++j) {
          oa[j] = ob[j] = gn[j] = make_float2(0.f, 0.f);
          if (8 * j >= prm.half) continue;
          if (la) oa[j] = *reinterpret_cast<const float2*>(xa + 8 * j);
          if (lb) ob[j] = *reinterpret_cast<const float2*>(xb + 8 * j);
          if (prm.gain != nullptr) gn[j] = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(prm.gain + f0 + 8 * j));
        }
        const bool ok = sums_ready();
        float v[U][4];
#pragma unroll
        for (int j = 0; j < U; ++j)
          if (8 * j < prm.half) ld_frag8(taddr + 8 * j, v[j]);
        ld_wait();
        float qa = 0.f, qb = 0.f;
#pragma unroll
        for (int j = 0; j < U; ++j) {
          if (8 * j >= prm.half) continue;
          if (!ok) v[j][0] = v[j][1] = v[j][2] = v[j][3] = 0.f;
          const float a0 = oa[j].x + v[j][0], a1 = oa[j].y + v[j][1], b0 = ob[j].x + v[j][2], b1 = ob[j].y + v[j][3];
          if (la) *reinterpret_cast<float2*>(xa + 8 * j) = make_float2(a0, a1);
          if (lb) *reinterpret_cast<float2*>(xb + 8 * j) = make_float2(b0, b1);
          if (prm.gain == nullptr) continue;
          if (la) *reinterpret_cast<uint32_t*>(prm.xn + (size_t)ra * prm.out + f0 + 8 * j) = pack2(gn[j].x * a0, gn[j].y * a1);
          if (lb) *reinterpret_cast<uint32_t*>(prm.xn + (size_t)rb * prm.out + f0 + 8 * j) = pack2(gn[j].x * b0, gn[j].y * b1);
          qa += a0 * a0 + a1 * a1;
          qb += b0 * b0 + b1 * b1;
        }
        if (prm.gain != nullptr) {
          qa += __shfl_xor_sync(0xffffffffu, qa, 1); qa += __shfl_xor_sync(0xffffffffu, qa, 2);
          qb += __shfl_xor_sync(0xffffffffu, qb, 1); qb += __shfl_xor_sync(0xffffffffu, qb, 2);
          if ((lane & 3) == 0 && la) prm.ss[(size_t)ra * prm.tiles_per_seg + lt] = qa;
          if ((lane & 3) == 0 && lb) prm.ss[(size_t)rb * prm.tiles_per_seg + lt] = qb;
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base_slot), "r"(prm.tmem_cols) : "memory");
  }
  if (threadIdx.x == 0 && abort_flag && prm.err_flag) *prm.err_flag = AMPH_ERR_TIMEOUT;
}

// K blocks per stage and shared memory of the forms.  Gate / up: one CTA per SM with everything: a launch of 180 MB is bound by the
// bytes it has in flight, so it took 34.0 us back to back with 126 KB, 31.8 with 170 and 30.9 with 215 (weights alone, neither
// activations nor MMAs: 28.6; 64-row tiles with two stages of 48 KB: 35.0).  The others have two CTAs per SM.
constexpr int kGateUpKb = 2, kQkvKb = 2, kResidKb = 4;
constexpr size_t kGateUpSmem = 215 * 1024, kTwoPerSm = 110 * 1024;

// Rings, tensor memory and everything else that does not depend on the epilogue; false: not covered.
bool rows_params(TcGemm* g, int xb, int n, int in, int rows, size_t smem_limit, int ks, int m, int accs, RowsMaps* maps, RowsParams* prm,
                 size_t* smem) {
  if (!g || xb < 0 || xb >= g->n_x || g->xcols[xb] != in || in % kTileK || rows < 1 || rows > m || n < 8 || n > 256 || n % (m / 8) || n * accs > 256) return false;
  memset(maps, 0, sizeof *maps);
  memset(prm, 0, sizeof *prm);
  prm->nt = (rows + 15) / 16 * 16;
  if (prm->nt > g->xrows[xb]) return false;
  prm->n = n;
  prm->rows = rows;
  prm->kblocks = prm->kb_cut = in / kTileK;
  if (accs == 2) prm->kb_cut = prm->kblocks / 2;
  const size_t x_stage = (size_t)ks * prm->nt * 128, w_stage = (size_t)ks * n * 128;
  int x_stages = m == 128 ? 4 : 3;                                  // one less where it would leave fewer than four of weights
  while (x_stages > 2 && 1024 + x_stages * x_stage + 4 * w_stage > smem_limit) --x_stages;
  const size_t x_ring = x_stages * x_stage;
  prm->x_stages = x_stages;
  int ws = smem_limit > 1024 + x_ring ? (int)((smem_limit - 1024 - x_ring) / w_stage) : 0;
  const int its = (prm->kblocks + ks - 1) / ks;
  if (ws > its) ws = its;
  if (ws > kMaxRing) ws = kMaxRing;
  if (ws < 2) ws = 2;
  prm->w_stages = ws;
  prm->l2_prefetch = 1;                              // 0 and 2: the same, 4: +0.5 % on a step
  prm->tmem_cols = 32;
  while (prm->tmem_cols < n * accs) prm->tmem_cols *= 2;
  *smem = 1024 + x_ring + ws * w_stage;
  const size_t floor = 1024 + x_ring + (size_t)m * 128;            // an MMA reads M rows from the last activation box on
  if (*smem < floor) *smem = floor;
  if (*smem > (size_t)g->max_smem - 2048) return false;
  const CUtensorMap* mx = g->get(g->xptr[xb], g->xrows[xb], in, prm->nt, ks);
  if (!mx) return false;
  maps->x = *mx;
  prm->err_flag = g->err_flag;
  prm->wait_limit_ns = g->wait_limit_ns;
  prm->extra_tx = g->extra_tx;
  return true;
}

template <int EPI, int KS, int M = 64>
bool rows_run(TcGemm* g, const RowsMaps& maps, const RowsParams& prm, int tiles, size_t smem, cudaStream_t st) {
  if (!g->rows_ready[M == 128 ? 3 : EPI]) {
    if (cudaFuncSetAttribute(tc_rows_kernel<EPI, KS, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, g->max_smem - 2048) != cudaSuccess) return false;
    g->rows_ready[M == 128 ? 3 : EPI] = true;
  }
  return launch_pdl(tc_rows_kernel<EPI, KS, M>, dim3(tiles), dim3(kRowsThreads), smem, st, maps, prm) == cudaSuccess;
}

}  // namespace

bool tc_rows_launch_swiglu(TcGemm* g, int xb, const void* w_gate, const void* w_up, int f, int in, int rows, void* act, const RowScale& rs,
                           cudaStream_t st) {
  if (!g || !w_gate || !w_up || !act || f % 64 || (((uintptr_t)w_gate | (uintptr_t)w_up) & 15)) return false;
  // Tiles of 64 rows of each matrix at two CTAs per SM (tc_gemm_kernel) stay where they are as fast or faster: for up to 16 rows,
  // whose activations leave their ring deep enough, and from 1.5 tiles per SM on, when tiles of up to 128 rows here leave too few
  // stages.  Us a launch, back to back, at 4096 x 2 x 11008: 16 rows 29.7, here 31.5; 32 rows 32.7 / 31.6; 64 rows 35.0 / 30.9.
  // A step's layer at 6656 x 2 x 17920: 2 % slower here.  Small matrices come here whatever the rows: more and shorter tiles.
  // More than 64 rows (contexts that keep one order of sums): in place of tc_gemm_launch's split-K sums and swiglu_kernel, where there
  // are at most two of them, bit for bit.  128 rows, 4096 x 2 x 11008 (7B, 2048 tokens of context, six steps): 28.6 ms with the two
  // kernels (37.9 + 4.5 us a layer), now 27.6.
  const bool m128 = rows > 64;
  const int accs = m128 ? tc_gemm_splits(g, 2 * (f / kTileM), in / kTileK, rows) : 1;
  if (m128 && (accs > 2 || f % kTileM || in / kTileK % accs)) return false;
  const int tiles64 = f / 64;
  if (tiles64 * 2 > g->sm_count && (rows <= 16 || tiles64 * 2 > 3 * g->sm_count)) return false;
  int half = ((f + g->sm_count - 1) / g->sm_count + 7) / 8 * 8;      // (M = 128 takes N in steps of 16)
  if (half > 128) half = 128;
  RowsMaps maps;
  RowsParams prm;
  size_t smem;
  if (!rows_params(g, xb, 2 * half, in, rows, kGateUpSmem, m128 ? 1 : kGateUpKb, m128 ? 128 : 64, accs, &maps, &prm, &smem)) return false;
  const bool up_first = (const char*)w_up < (const char*)w_gate;
  const uint64_t gap = up_first ? (const char*)w_gate - (const char*)w_up : (const char*)w_up - (const char*)w_gate;
  const CUtensorMap* m = g->get_halves(up_first ? w_up : w_gate, gap, f, in, half, m128 ? 1 : kGateUpKb);
  if (!m) return false;
  maps.w[0] = *m;
  prm.half = half;
  prm.tiles_per_seg = (f + half - 1) / half;
  prm.act = (__nv_bfloat16*)act;
  prm.f = f;
  prm.up_first = up_first ? 1 : 0;
  prm.rs = rs;
  if (m128) return rows_run<ROWS_SWIGLU, 1, 128>(g, maps, prm, prm.tiles_per_seg, smem, st);
  return rows_run<ROWS_SWIGLU, kGateUpKb>(g, maps, prm, prm.tiles_per_seg, smem, st);
}

bool tc_rows_launch_qkv_rope(TcGemm* g, int xb, const void* wq, const void* wk, const void* wv, int n_heads, int dh, int in, int rows, void* q,
                             KvView kv, const RowMeta* meta, const float2* rope, int max_ctx, const RowScale& rs, cudaStream_t st) {
  if (!g || !wq || !wk || !wv || !q || !kv.k || !kv.v || !meta || !rope || (dh != 64 && dh != 128)) return false;
  if (((uintptr_t)wq | (uintptr_t)wk | (uintptr_t)wv) & 15) return false;
  const int d = n_heads * dh;
  // Up to 32 rows tc_gemm_kernel's 64-row tiles, from 2/5 of a wave of them on: us a step of 8 layers there / here, 16 rows, width 512
  // 258.5 / 253.4, 768 295 / 292, 1024 312 / 313, 1280 333 / 343, 1536 368 / 373, 2048 430 / 442; 32 rows, width 1280 340 / 350, 2048
  // 447 / 457.  Above 32 rows here: 4096 x 3 x 4096 back to back, 48 rows 21.2 / 19.9, 64 rows 21.7 / 20.7; a pass of 8 steps x 8 layers,
  // 48 rows 9780 / 9660, 64 rows 10097 / 9963, at 6656 (6 layers x 6 steps) 14036 / 13767.
  if (rows <= 32 && 3 * d / 64 * 5 > 2 * g->sm_count) return false;
  int half = 8;                                      // the smallest tile that leaves all CTAs resident at once
  while (half < dh / 2 && 3 * d / 2 / half > 2 * g->sm_count) half *= 2;
  RowsMaps maps;
  RowsParams prm;
  size_t smem;
  if (!rows_params(g, xb, 2 * half, in, rows, kTwoPerSm, kQkvKb, 64, 1, &maps, &prm, &smem)) return false;
  const void* w[3] = {wq, wk, wv};
  for (int s = 0; s < 3; ++s) {
    const CUtensorMap* m = g->get_halves(w[s], (uint64_t)(dh / 2) * in * 2, d, in, half, kQkvKb);
    if (!m) return false;
    maps.w[s] = *m;
  }
  prm.half = half;
  prm.tiles_per_seg = d / 2 / half;
  prm.rs = rs;
  prm.q = (__nv_bfloat16*)q;
  prm.kc = (__nv_bfloat16*)kv.k;
  prm.vc = (__nv_bfloat16*)kv.v;
  prm.meta = meta;
  prm.rope = rope;
  prm.n_heads = n_heads;
  prm.dh = dh;
  prm.max_ctx = max_ctx;
  return rows_run<ROWS_ROPE, kQkvKb>(g, maps, prm, 3 * prm.tiles_per_seg, smem, st);
}

bool tc_rows_launch_resid(TcGemm* g, int xb, const void* w, int out, int in, int rows, float* x, const void* gain, void* xn, float* ss,
                          int* cols, cudaStream_t st) {
  if (!g || !w || !x || ((uintptr_t)w & 15) || (gain && (!xn || !ss))) return false;
  // Without split-K every CTA reads all activation rows for a tile of 16 features, so only where both sides are short.  Us a step of
  // 8 layers, 16 / 32 / 64 rows, with split-K sums and a kernel that adds them | with this: width 1280 347 / 360 / 370 | 346 / 353 / 361,
  // 1536 378 / 389 / 400 | 375 / 387 / 395, 2048 432 / 450 / 465 | 444 / 458 / 464; the down projection alone, 2048 -> 1024 303 / 320 / 318 |
  // 307 / 309 / 310, 2048 -> 768 292 / 299 / 304 | 282 / 290 / 289; a launch at 4096 x 4096 (16 rows) 11.6 us against 7.3 + 3.0.
  if (out > kRowsResidOut || in > kRowsResidMax || out % 16) return false;
  const int half = 16;
  RowsMaps maps;
  RowsParams prm;
  size_t smem;
  if (!rows_params(g, xb, half, in, rows, kTwoPerSm, kResidKb, 64, 1, &maps, &prm, &smem)) return false;
  const CUtensorMap* m = g->get(w, out, in, half, kResidKb);
  if (!m) return false;
  maps.w[0] = *m;
  prm.half = half;
  prm.tiles_per_seg = out / half;
  prm.x = x;
  prm.gain = (const __nv_bfloat16*)gain;
  prm.xn = (__nv_bfloat16*)xn;
  prm.ss = ss;
  prm.out = out;
  *cols = half;
  return rows_run<ROWS_RESID, kResidKb>(g, maps, prm, prm.tiles_per_seg, smem, st);
}

}  // namespace amph
