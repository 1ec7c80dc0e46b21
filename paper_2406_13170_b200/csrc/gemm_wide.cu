// bf16 projection for many activation rows (up to 512) on CTA pairs:  Y^T[out][rows] = W[out][in] . X^T.
//
// A cluster of two CTAs owns 256 weight rows and a block of up to 256 activation rows: one tcgen05.mma.cta_group::2 (M = 256,
// N <= 256) per 16 columns of K.  Each CTA stages its own 128 weight rows and HALF of the activation rows: 32 KB per 64
// columns of K at N = 256, i.e. 64 bytes of L2 -> SM traffic per clock of MMA, against 80 with one CTA per 128 weight rows and
// 512 activation rows (which made L2 the bound).  With 257..512 rows two neighbouring pairs take the two row blocks of the
// same weights at the same time, so weights still cross HBM once.  Tensor memory holds two accumulators: the epilogue of
// one piece of work runs under the main loop of the next.
//
// Balance: a launch is `tiles` x K work.  Cut tile by tile, 48 tiles (q / k / v at d = 4096) keep 65 % of the 74 pairs busy and
// 86 (gate / up) take two waves of 58 %.  So group g of pairs (a pair per row block) takes the g-th of equal ranges of the
// (tile, K) line: a range may begin inside a tile (its first segment then leaves fp32 partial sums in scratch and raises a
// flag) and may end inside one (the pair that holds a tile's first K columns waits for the flags of the groups after it, adds
// their sums in order and runs the epilogue).  A flag is raised before its pair waits for anybody, and pairs are numbered
// against the launch order, so a pair only ever waits for pairs that became resident before it; the wait is bounded all the
// same.  Where the consumer adds split-K sums anyway (output and down projections) the K ranges are cut evenly per tile.
//
// Warp roles: 0 = TMA producer, 1 = MMA issuer (of the even CTA), 2-9 = epilogue (two warps per TMEM lane quarter).
#include "gemm_tc_common.cuh"

namespace amph {

using namespace tc;

namespace {

constexpr int kWideThreads = 320;
constexpr int kEpiThreads = 256;
constexpr int kUnitKb = 2;            // K blocks per unit of work: ranges are cut at multiples of 128 columns
constexpr int kMaxWideRows = 512;
constexpr int kMaxStages = 8;

struct WideMaps {
  CUtensorMap w[kMaxSeg];
  CUtensorMap x;
};

enum { WIDE_PLAIN = 0, WIDE_SWIGLU = 1, WIDE_ROPE = 2 };

struct WideParams {
  int tiles_per_seg, tiles;
  int kblocks, units_per_tile;
  int splits;               // 0: equal ranges of all work (fix-up through scratch); > 0: K ranges per tile, one per group
  int groups, nrb;          // groups of nrb pairs (row blocks)
  int n;                    // activation rows per MMA (a multiple of 32)
  int tmem_cols;
  int rows, stages;
  float* P;                 // PLAIN: P[split][row][feature]
  size_t split_stride;
  int ld;
  float* scratch;           // [pair][cta][chunk of 16 rows][row quad][128 features] float4: partial sums of a pair's first segment
  int* flags;               // [pair][cta]; zero between launches (whoever consumes a flag lowers it)
  __nv_bfloat16* act;       // SWIGLU
  int f, up_first;
  RowScale rs;
  __nv_bfloat16* q;         // ROPE
  RopeGroups gr;
  int n_heads, dh, max_ctx;
  int* err_flag;
  unsigned long long wait_limit_ns;
};

struct Segment { int tile, kb0, kb1; };

// The segments of one group's range of work units, in order.
struct SegIter {
  int u, end, upt, kblocks;
  __device__ bool next(Segment& s) {
    if (u >= end) return false;
    const int t = u / upt, a = u - t * upt;
    int e = end - t * upt;
    if (e > upt) e = upt;
    s.tile = t;
    s.kb0 = a * kUnitKb;
    s.kb1 = e * kUnitKb < kblocks ? e * kUnitKb : kblocks;
    u = t * upt + e;
    return true;
  }
};

// First work unit of a group; range_begin(group + 1) is its end.
__device__ __forceinline__ int range_begin(const WideParams& prm, int group) {
  if (prm.splits > 0) {
    const int t = group / prm.splits, s = group - t * prm.splits;
    return t * prm.units_per_tile + s * prm.units_per_tile / prm.splits;
  }
  return (int)((long long)group * prm.tiles * prm.units_per_tile / prm.groups);
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// Copies of a CTA pair: the destination is this CTA's shared memory, the barrier the even CTA's.
__device__ __forceinline__ void tma_pair_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_pair_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void tma_pair_4d(void* dst, const CUtensorMap* map, int x, int y, int z, int w, uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5}], [%6], %7;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void tma_pair_5d(void* dst, const CUtensorMap* map, int x, int y, int z, int w, int v, uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3, %4, %5, %6}], [%7], %8;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(v), "r"(bar), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
// Arrives at the same barrier of both CTAs once the MMAs issued so far are complete.
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
        "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// Rows of a tile, in both fused forms: 16 rows of one kind, then the 16 rows they are combined with (gate / up, or the two
// members of 16 rotation pairs), four times over.  Lanes l and l + 16 of an epilogue warp then hold the two operands of one
// output feature for 16 activation rows; after one exchange lane l < 16 has both for the first eight rows, lane l + 16 for
// the other eight, and half a warp writes 16 neighbouring features (32 bytes) of a row.
__device__ __forceinline__ void pair_up(const float* v, int lane, float* first, float* second) {
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float got = __shfl_xor_sync(0xffffffffu, lane < 16 ? v[8 + j] : v[j], 16);
    first[j] = lane < 16 ? v[j] : got;
    second[j] = lane < 16 ? got : v[8 + j];
  }
}

template <int EPI>
__global__ void __launch_bounds__(kWideThreads, 1)
tc_wide_kernel(const __grid_constant__ WideMaps maps, const WideParams prm) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ float inv_s[EPI == WIDE_PLAIN ? 1 : 256];             // 1 / rms of this pair's activation rows
  __shared__ int slot_s[EPI == WIDE_ROPE ? 256 : 1];               // cache slot of a row, -1: not stored
  __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], accum_full[2], accum_empty[2];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;

  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int pair = prm.groups * prm.nrb - 1 - (int)(blockIdx.x >> 1);        // against the launch order (see above)
  const int group = pair / prm.nrb, rb = pair - group * prm.nrb;
  const int stages = prm.stages, n = prm.n;
  const uint32_t b_tile = (uint32_t)n / 2 * 128, a_tile = kTileM * 128;
  const uint32_t stage_bytes = a_tile + b_tile;
  const unsigned long long limit_ns = prm.wait_limit_ns;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const SegIter first = {range_begin(prm, group), range_begin(prm, group + 1), prm.units_per_tile, prm.kblocks};

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&accum_full[s], 1); mbar_init(&accum_empty[s], 2 * kEpiThreads / 32); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(prm.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync_all();                                                // both CTAs' barriers exist before any copy or MMA signals them
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_d = tmem_base_slot;

  if (warp == 0) {
    // ---------------- TMA producer of this CTA's half of the operands
    const bool leader = elect_one();
    const uint64_t wpol = l2_evict_first_policy();
    auto load_w = [&](int st, const Segment& s, int kb) {
      const int seg = s.tile / prm.tiles_per_seg, lt = s.tile - seg * prm.tiles_per_seg;
      const uint32_t bar = map_to_rank(smem_u32(&full_bar[st]), 0);
      uint8_t* dst = smem + (size_t)st * stage_bytes;
      if (rank == 0) mbar_expect_tx(&full_bar[st], 2 * stage_bytes);
      if (EPI == WIDE_SWIGLU) tma_pair_4d(dst, &maps.w[0], kb * kTileK, 0, 0, (lt * 2 + (int)rank) * 4, bar, wpol);
      else if (EPI == WIDE_ROPE) tma_pair_5d(dst, &maps.w[seg], kb * kTileK, 0, 0, 0, (lt * 2 + (int)rank) * kTileM / prm.dh, bar, wpol);
      else tma_pair_3d(dst, &maps.w[seg], 0, (lt * 2 + (int)rank) * kTileM, kb, bar, wpol);
    };
    auto load_x = [&](int st, int kb) {
      const uint32_t bar = map_to_rank(smem_u32(&full_bar[st]), 0);
      tma_pair_3d(smem + (size_t)st * stage_bytes + a_tile, &maps.x, 0, rb * n + (int)rank * (n / 2), kb, bar);
    };
    // weights do not depend on the kernel before: fill the ring with them, then wait, then fetch those stages' activations
    SegIter it = first;
    Segment sg;
    bool have = it.next(sg);
    int kb = have ? sg.kb0 : 0, i = 0;
    for (; i < stages && have; ++i) {
      if (leader) load_w(i, sg, kb);
      if (++kb == sg.kb1) { have = it.next(sg); kb = sg.kb0; }
    }
    __syncwarp();
    pdl_wait();
    {
      SegIter bt = first;
      Segment bs;
      bool more = bt.next(bs);
      int bk = more ? bs.kb0 : 0;
      for (int j = 0; j < i; ++j) {
        if (leader) load_x(j, bk);
        if (++bk == bs.kb1) { more = bt.next(bs); bk = bs.kb0; }
      }
    }
    __syncwarp();
    for (; have; ++i) {
      const int st = i % stages, round = i / stages;
      if (!__all_sync(0xffffffffu, mbar_wait(&empty_bar[st], (round & 1) ^ 1, &abort_flag, limit_ns))) break;
      if (leader) { load_w(st, sg, kb); load_x(st, kb); }
      __syncwarp();
      if (++kb == sg.kb1) { have = it.next(sg); kb = sg.kb0; }
    }
    if (abort_flag && rank == 0 && lane == 0) {          // drain: both CTAs' copies signal the even CTA's barriers
      const unsigned long long t0 = now_ns();
      for (int j = i > stages ? i - stages : 0; j < i; ++j)
        while (!mbar_try(&full_bar[j % stages], (j / stages) & 1) && now_ns() - t0 < limit_ns) {}
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (even CTA)
    if (rank == 0) {
      const bool leader = elect_one();
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      SegIter it = first;
      Segment sg;
      bool ok = true;
      int i = 0;
      for (int j = 0; ok && it.next(sg); ++j) {
        const int as = j & 1, around = j >> 1;
        if (around > 0) ok = __all_sync(0xffffffffu, mbar_wait(&accum_empty[as], (around & 1) ^ 1, &abort_flag, limit_ns));
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d = tmem_d + (uint32_t)(as * n);
        for (int kb = sg.kb0; ok && kb < sg.kb1; ++kb, ++i) {
          const int st = i % stages;
          ok = __all_sync(0xffffffffu, mbar_wait(&full_bar[st], (i / stages) & 1, &abort_flag, limit_ns));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (leader) {
            const uint32_t a_addr = smem_u32(smem + (size_t)st * stage_bytes);
            const uint64_t ad = umma_desc(a_addr), bd = umma_desc(a_addr + a_tile);
#pragma unroll
            for (int k = 0; k < kTileK / kUmmaK; ++k)
              umma_pair(d, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), idesc, kb > sg.kb0 || k > 0 ? 1u : 0u);
            umma_commit_pair(&empty_bar[st]);
          }
          __syncwarp();
        }
        if (ok && leader) umma_commit_pair(&accum_full[as]);
        __syncwarp();
      }
    }
  } else {
    // ---------------- epilogue
    const int quarter = warp & 3, half = (warp - 2) >> 2, et = threadIdx.x - 64;
    const int chunks = n / 16;                           // chunks of 16 activation rows
    const int row0 = rb * n, my_rows = prm.rows - row0 < n ? prm.rows - row0 : n;
    pdl_wait();
    if constexpr (EPI != WIDE_PLAIN) {
      if (et < my_rows) inv_s[et] = row_scale(prm.rs, row0 + et);
    }
    if constexpr (EPI == WIDE_ROPE) {
      if (et < my_rows) {
        const int g = (row0 + et) / prm.gr.rpg, rl = row0 + et - g * prm.gr.rpg;
        const RowMeta* meta = prm.gr.meta[g];
        const int slot = meta->slot[rl];
        slot_s[et] = rl < meta->n_rows && slot >= 0 && slot < prm.max_ctx ? slot : -1;
      }
    }
    epi_sync();
    const size_t slot_quads = (size_t)chunks * 4 * kTileM;           // float4s of one CTA's partial sums
    const int frow = quarter * 32 + lane;                // row of this CTA's tile
    float4* const scratch = reinterpret_cast<float4*>(prm.scratch) + frow;
    SegIter it = first;
    Segment sg;
    for (int j = 0; it.next(sg); ++j) {
      const int as = j & 1;
      bool ok = __all_sync(0xffffffffu, mbar_wait(&accum_full[as], (j >> 1) & 1, &abort_flag, limit_ns));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t t0 = tmem_d + (uint32_t)(as * n) + ((uint32_t)(quarter * 32) << 16);
      if (prm.splits == 0 && sg.kb0 > 0) {               // not the tile's first K columns: leave the sums to the pair that has them
        float4* dst = scratch + ((size_t)pair * 2 + rank) * slot_quads;
        for (int c = half; c < chunks; c += 2) {
          uint32_t v[16];
          tmem_ld16(t0 + (uint32_t)c * 16, v);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int e = 0; e < 4; ++e)
            __stcg(dst + (size_t)(c * 4 + e) * kTileM,
                   ok ? make_float4(__uint_as_float(v[4 * e]), __uint_as_float(v[4 * e + 1]), __uint_as_float(v[4 * e + 2]), __uint_as_float(v[4 * e + 3]))
                      : make_float4(0.f, 0.f, 0.f, 0.f));
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&accum_empty[as]), 0));
        __threadfence();
        epi_sync();
        if (et == 0) asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(prm.flags + pair * 2 + rank), "r"(1) : "memory");
        continue;
      }
      int helpers = 0;                                    // groups after this one that hold the rest of the tile
      if (prm.splits == 0 && sg.kb1 < prm.kblocks) {
        const int tile_end = (sg.tile + 1) * prm.units_per_tile;
        while (group + 1 + helpers < prm.groups && range_begin(prm, group + 1 + helpers) < tile_end) ++helpers;
        if (et < helpers) {
          const int* flag = prm.flags + (pair + (1 + et) * prm.nrb) * 2 + rank;
          const unsigned long long w0 = now_ns();
          for (uint32_t w = 1;; ++w) {
            int up;
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(up) : "l"(flag) : "memory");
            if (up) break;
            if ((w & 63u) == 0u && (*(volatile int*)&abort_flag || now_ns() - w0 > limit_ns)) { abort_flag = 1; break; }
          }
        }
        epi_sync();
        ok = ok && *(volatile int*)&abort_flag == 0;
      }
      const int seg = sg.tile / prm.tiles_per_seg, lt = sg.tile - seg * prm.tiles_per_seg;
      const float4* src = scratch + ((size_t)(pair + prm.nrb) * 2 + rank) * slot_quads;
      const size_t next_helper = (size_t)prm.nrb * 2 * slot_quads;
      const int gph = prm.dh >> 5, hdim = prm.dh >> 1;                    // ROPE: groups of 16 pairs per head
      for (int c = half; c < chunks; c += 2) {
        const int r0 = c * 16;                            // first activation row of the chunk, within this pair's block
        if (r0 >= my_rows) break;
        const int rl8 = r0 + (lane >> 4) * 8;             // first of the eight rows this lane finishes (fused forms)
        // every load of the chunk is in flight before the first use
        float4 o[4];
        if (helpers > 0) {
#pragma unroll
          for (int e = 0; e < 4; ++e) o[e] = __ldcg(src + (size_t)(c * 4 + e) * kTileM);
        }
        float2 cs[8];
        int g = 0, i0 = 0;
        if constexpr (EPI == WIDE_ROPE) {
          g = (row0 + r0) / prm.gr.rpg;                   // a group's height is a multiple of 16
          i0 = (quarter % gph) * 16 + (lane & 15);
          if (seg < 2) {
            const float2* table = prm.gr.rope[g] + (size_t)(row0 + rl8 - g * prm.gr.rpg) * hdim + i0;
#pragma unroll
            for (int e = 0; e < 8; ++e) cs[e] = table[e * hdim];
          } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) cs[e] = make_float2(1.f, 0.f);
          }
        }
        uint32_t raw[16];
        tmem_ld16(t0 + (uint32_t)r0, raw);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        float v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) v[e] = ok ? __uint_as_float(raw[e]) : 0.f;
        for (int hp = 0; hp < helpers; ++hp) {
#pragma unroll
          for (int e = 0; e < 4; ++e) { v[4 * e] += o[e].x; v[4 * e + 1] += o[e].y; v[4 * e + 2] += o[e].z; v[4 * e + 3] += o[e].w; }
          if (hp + 1 < helpers) {
#pragma unroll
            for (int e = 0; e < 4; ++e) o[e] = __ldcg(src + (hp + 1) * next_helper + (size_t)(c * 4 + e) * kTileM);
          }
        }
        if constexpr (EPI == WIDE_PLAIN) {
          const int split = prm.splits > 0 ? group % prm.splits : 0;
          float* out = prm.P + (size_t)split * prm.split_stride + (size_t)(row0 + r0) * prm.ld + (size_t)sg.tile * 256 + rank * kTileM + frow;
#pragma unroll
          for (int e = 0; e < 16; ++e)
            if (r0 + e < my_rows) out[(size_t)e * prm.ld] = v[e];
        } else {
          float x0[8], x1[8];
          pair_up(v, lane, x0, x1);
          if constexpr (EPI == WIDE_SWIGLU) {
            __nv_bfloat16* out = prm.act + (size_t)(row0 + rl8) * prm.f + (lt * 2 + (int)rank) * 64 + quarter * 16 + (lane & 15);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              if (rl8 + e < my_rows) {
                const float sc = inv_s[rl8 + e];
                const float t = (prm.up_first ? x1[e] : x0[e]) * sc, u = (prm.up_first ? x0[e] : x1[e]) * sc;
                out[(size_t)e * prm.f] = __float2bfloat16(__fdividef(t, 1.0f + __expf(-t)) * u);
              }
            }
          } else {
            const int head = (lt * 2 + (int)rank) * kTileM / prm.dh + quarter / gph;
            __nv_bfloat16* cache = (__nv_bfloat16*)(seg == 1 ? prm.gr.kc[g] : prm.gr.vc[g]) + (size_t)head * prm.max_ctx * prm.dh + i0;
            __nv_bfloat16* qrow = prm.q + (size_t)(row0 + rl8) * prm.n_heads * prm.dh + head * prm.dh + i0;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              if (rl8 + e >= my_rows) continue;
              const float sc = inv_s[rl8 + e];
              const float lo = x0[e] * sc, hi = x1[e] * sc;
              __nv_bfloat16* dst = qrow + (size_t)e * prm.n_heads * prm.dh;
              if (seg > 0) {
                const int slot = slot_s[rl8 + e];
                dst = slot >= 0 ? cache + (size_t)slot * prm.dh : nullptr;
              }
              if (dst != nullptr) {
                dst[0] = __float2bfloat16(lo * cs[e].x - hi * cs[e].y);
                dst[hdim] = __float2bfloat16(hi * cs[e].x + lo * cs[e].y);
              }
            }
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&accum_empty[as]), 0));
      if (helpers > 0) {                                  // every thread has read the sums: lower the flags for the next launch
        epi_sync();
        if (et < helpers) prm.flags[(pair + (1 + et) * prm.nrb) * 2 + rank] = 0;
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync_all();                                     // no CTA leaves while its partner may still signal or read its shared memory
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(prm.tmem_cols) : "memory");
  }
  if (threadIdx.x == 0 && abort_flag && prm.err_flag) *prm.err_flag = AMPH_ERR_TIMEOUT;
}

constexpr size_t kWideSmem = 221 * 1024;                  // ring + alignment; the static part needs up to 3 KB of the 227

// Everything of a launch that does not depend on the epilogue; false: the shape is not covered.
bool wide_params(TcGemm* g, int xb, int n_seg, int tiles_per_seg, int in, int rows, int splits, float* scratch_end, size_t scratch_floats,
                 WideMaps* maps, WideParams* prm) {
  if (!g || g->wide_pairs < 2 || xb < 0 || xb >= g->n_x || g->xcols[xb] != in) return false;
  if (in % kTileK || rows < 32 || rows > kMaxWideRows || rows > g->xrows[xb] || n_seg < 1 || n_seg > kMaxSeg) return false;
  memset(maps, 0, sizeof *maps);
  memset(prm, 0, sizeof *prm);
  prm->nrb = rows > 256 ? 2 : 1;
  prm->n = ((rows + prm->nrb - 1) / prm->nrb + 31) / 32 * 32;        // an M = 256 pair MMA takes N in steps of 32
  const CUtensorMap* mx = g->get(g->xptr[xb], g->xrows[xb], in, prm->n / 2, 1);
  if (!mx) return false;
  maps->x = *mx;
  prm->tmem_cols = 64;
  while (prm->tmem_cols < 2 * prm->n) prm->tmem_cols *= 2;
  prm->tiles_per_seg = tiles_per_seg;
  prm->tiles = n_seg * tiles_per_seg;
  prm->kblocks = in / kTileK;
  prm->units_per_tile = (prm->kblocks + kUnitKb - 1) / kUnitKb;
  prm->splits = splits;
  prm->groups = g->wide_pairs / prm->nrb;
  const int units = prm->tiles * prm->units_per_tile;
  if (splits > 0) {
    if (splits > prm->units_per_tile) return false;
    prm->groups = prm->tiles * splits;
  } else {
    // at least four units (512 columns) a group, unless there are more tiles than that; no more pairs than scratch
    const int most = units / 4 > prm->tiles ? units / 4 : prm->tiles;
    if (prm->groups > most) prm->groups = most;
    const size_t per_group = (size_t)prm->nrb * 2 * prm->n * kTileM;
    if ((size_t)prm->groups > scratch_floats / per_group) prm->groups = (int)(scratch_floats / per_group);
    if (prm->groups < 1 || !scratch_end || !g->wide_flags || 2 * prm->groups * prm->nrb > kWideFlags) return false;
    prm->scratch = scratch_end - (size_t)prm->groups * per_group;    // the buffer's end: its beginning may hold the result
  }
  prm->rows = rows;
  const size_t stage = (size_t)kTileM * 128 + (size_t)prm->n / 2 * 128;
  prm->stages = (int)((kWideSmem - 1024) / stage);
  if (prm->stages > kMaxStages) prm->stages = kMaxStages;
  prm->flags = g->wide_flags;
  prm->err_flag = g->err_flag;
  prm->wait_limit_ns = g->wait_limit_ns;
  return true;
}

template <int EPI>
bool wide_run(const WideMaps& maps, const WideParams& prm, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * prm.groups * prm.nrb);
  cfg.blockDim = dim3(kWideThreads);
  cfg.dynamicSmemBytes = kWideSmem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = 2;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, tc_wide_kernel<EPI>, maps, prm) == cudaSuccess;
}

}  // namespace

void tc_wide_init(TcGemm* g) {
  g->wide_pairs = 0;
  if ((size_t)g->max_smem < kWideSmem + 4 * 1024) return;
  int clusters = 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g->sm_count / 2 * 2);
  cfg.blockDim = dim3(kWideThreads);
  cfg.dynamicSmemBytes = kWideSmem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cudaFuncSetAttribute(tc_wide_kernel<WIDE_PLAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWideSmem) != cudaSuccess ||
      cudaFuncSetAttribute(tc_wide_kernel<WIDE_SWIGLU>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWideSmem) != cudaSuccess ||
      cudaFuncSetAttribute(tc_wide_kernel<WIDE_ROPE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWideSmem) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&clusters, tc_wide_kernel<WIDE_ROPE>, &cfg) != cudaSuccess || clusters < 1) {
    cudaGetLastError();
    return;
  }
  g->wide_pairs = clusters < g->sm_count / 2 ? clusters : g->sm_count / 2;
}

void tc_wide_bind(TcGemm* g, float* scratch, size_t scratch_floats, int* flags) {
  g->wide_scratch = scratch;
  g->wide_scratch_floats = scratch_floats / 64 * 64;
  g->wide_flags = flags;
}

bool tc_wide_launch(TcGemm* g, int xb, const void* const* w, int n_seg, int out, int in, int rows, float* P, size_t p_floats,
                    int* splits_out, size_t* split_stride, cudaStream_t st) {
  if (!g || g->wide_pairs < 2 || out % 256 || in % kTileK) return false;
  const int tiles = n_seg * (out / 256), units = (in / kTileK + kUnitKb - 1) / kUnitKb;
  const size_t ld = (size_t)n_seg * out, stride = (size_t)rows * ld;
  if (stride > p_floats) return false;
  // Few tiles: the consumer adds the K ranges' sums (one per group).  Many: equal ranges of all the work, one sum.
  int splits = 0;
  const int groups = g->wide_pairs / (rows > 256 ? 2 : 1);
  if (tiles * 2 <= groups || !g->wide_flags) {
    splits = groups / tiles;
    if (splits > units / 2) splits = units / 2;            // at least four K blocks per pair
    if (splits > 16) splits = 16;
    while (splits > 1 && splits * stride > p_floats) --splits;
    if (splits < 1) splits = 1;
  }
  WideMaps maps;
  WideParams prm;
  // a cut tile's sums go to the end of the caller's buffer, behind the result
  const size_t end = p_floats / 64 * 64, used = (stride + 63) / 64 * 64;
  if (!wide_params(g, xb, n_seg, out / 256, in, rows, splits, P + end, end > used ? end - used : 0, &maps, &prm)) return false;
  for (int s = 0; s < n_seg; ++s) {
    if ((uintptr_t)w[s] & 15) return false;
    const CUtensorMap* m = g->get(w[s], out, in, kTileM, 1);
    if (!m) return false;
    maps.w[s] = *m;
  }
  prm.P = P;
  prm.ld = (int)ld;
  prm.split_stride = stride;
  if (!wide_run<WIDE_PLAIN>(maps, prm, st)) return false;
  *splits_out = splits > 0 ? splits : 1;
  *split_stride = stride;
  return true;
}

bool tc_wide_launch_swiglu(TcGemm* g, int xb, const void* w_gate, const void* w_up, int f, int in, int rows, void* act, const RowScale& rs,
                           cudaStream_t st) {
  if (!g || !g->wide_scratch || !w_gate || !w_up || !act || f % 128 || (((uintptr_t)w_gate | (uintptr_t)w_up) & 15)) return false;
  WideMaps maps;
  WideParams prm;
  if (!wide_params(g, xb, 1, f / 128, in, rows, 0, g->wide_scratch + g->wide_scratch_floats, g->wide_scratch_floats, &maps, &prm)) return false;
  const bool up_first = (const char*)w_up < (const char*)w_gate;
  const CUtensorMap* m = g->get_wide_pair(up_first ? w_up : w_gate, up_first ? w_gate : w_up, f, in);
  if (!m) return false;
  maps.w[0] = *m;
  prm.act = (__nv_bfloat16*)act;
  prm.f = f;
  prm.up_first = up_first ? 1 : 0;
  prm.rs = rs;
  return wide_run<WIDE_SWIGLU>(maps, prm, st);
}

bool tc_wide_launch_qkv_rope(TcGemm* g, int xb, const void* wq, const void* wk, const void* wv, int n_heads, int dh, int in, int rows, void* q,
                             const RopeGroups& gr, int max_ctx, const RowScale& rs, cudaStream_t st) {
  const int d = n_heads * dh;
  if (!g || !g->wide_scratch || !wq || !wk || !wv || !q || (dh != 64 && dh != 128) || d % 256 || gr.rpg % 16) return false;
  if (((uintptr_t)wq | (uintptr_t)wk | (uintptr_t)wv) & 15) return false;
  WideMaps maps;
  WideParams prm;
  if (!wide_params(g, xb, 3, d / 256, in, rows, 0, g->wide_scratch + g->wide_scratch_floats, g->wide_scratch_floats, &maps, &prm)) return false;
  const void* w[3] = {wq, wk, wv};
  for (int s = 0; s < 3; ++s) {
    const CUtensorMap* m = g->get_wide_rope(w[s], n_heads, dh, in);
    if (!m) return false;
    maps.w[s] = *m;
  }
  prm.q = (__nv_bfloat16*)q;
  prm.gr = gr;
  prm.n_heads = n_heads;
  prm.dh = dh;
  prm.max_ctx = max_ctx;
  prm.rs = rs;
  return wide_run<WIDE_ROPE>(maps, prm, st);
}

}  // namespace amph
