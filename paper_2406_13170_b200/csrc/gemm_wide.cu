// bf16 projection for many activation rows (up to 512) on CTA pairs:  Y^T[out][rows] = W[out][in] . X^T.
//
// A cluster of two CTAs owns 256 weight rows and a block of up to 256 activation rows: one tcgen05.mma.cta_group::2 (M = 256,
// N <= 256) per 16 columns of K.  Each CTA stages its own 128 weight rows and HALF of the activation rows: 32 KB per 64
// columns of K at N = 256, i.e. 64 bytes of L2 -> SM traffic per clock of MMA, against 80 with one CTA per 128 weight rows and
// 512 activation rows (which made L2 the bound).  A stage holds one or two K blocks (see unit_kb; the producers' and the
// issuer's loops must not divide for one block, 512 clocks of MMA at N = 256, to be enough: see below).
// With 257..512 rows two neighbouring pairs take the two row blocks of the same weights at the same time, so weights still
// cross HBM once.  Tensor memory holds two accumulators: the epilogue of one piece of work runs under the next main loop.
//
// Balance: a launch is `tiles` x K work.  Cut tile by tile, 48 tiles (q / k / v at d = 4096) keep 65 % of the 74 pairs busy and
// 86 (gate / up) take two waves of 58 %.  So group g of pairs (a pair per row block) takes the g-th of equal ranges of the
// (tile, K) line: a range may begin inside a tile (its first segment then leaves fp32 partial sums in scratch and raises a
// flag) and may end inside one (the pair that holds a tile's first K columns waits for the flags of the groups after it, adds
// their sums in order and runs the epilogue).  A flag is raised before its pair waits for anybody, and pairs are numbered
// against the launch order, so a pair only ever waits for pairs that became resident before it; the wait is bounded all the
// same.  Where the consumer adds split-K sums anyway the K ranges are cut evenly per tile.
//
// Output and down projection (WIDE_RESID) have few tiles (16 at d = 4096), so several pairs share one along K and all of them
// finish it: the pairs of a tile form a cluster, each gets a share of the tile's rows from the others by bulk copies through
// distributed shared memory, adds them in K order and applies the residual update.  Through global memory instead (sums
// written, a second kernel that adds them) d = 4096 / d_ffn = 11008 took, mean of the two: 128 rows 15.2 + 2.9 us, now 18.1; 256
// rows 20.9 + 5.6, now 27.0; 512 rows 28.0 + 8.8, now 31.8.  The projection behind it, whose ring fills while this one drains,
// starts 1-2 us earlier as well: a prefill of 512 rows took 8.80 ms, now 8.43, a batch of 8 x 40 nodes 90.2 ms, now 87.5.
//
// Warp roles: 0 = TMA producer, 1 = MMA issuer (of the even CTA), 2-17 = epilogue.
#include "gemm_tc_common.cuh"

namespace amph {

using namespace tc;

namespace {

constexpr int kEpiThreads = 512;      // four warps per TMEM lane quarter
constexpr int kWideThreads = 64 + kEpiThreads;
constexpr int kMaxWideRows = 512;
constexpr int kMaxStages = 8;
constexpr int kMaxGroups = kWideFlags / 2;

struct WideMaps {
  CUtensorMap w[kMaxSeg];
  CUtensorMap x;
};

enum { WIDE_PLAIN = 0, WIDE_SWIGLU = 1, WIDE_ROPE = 2, WIDE_RESID = 3 };

struct WideParams {
  int tiles_per_seg, tiles;
  int kblocks, units_per_tile;
  int kb;                   // K blocks per pipeline stage = unit of work: ranges are cut at multiples of 64 kb columns
  int splits;               // 0: equal ranges of all work (fix-up through scratch); > 0: K ranges per tile, one per group
  int groups, nrb;          // groups of nrb pairs (row blocks)
  int range[kMaxGroups + 1];   // splits == 0: first work unit of every group, and the end
  int n;                    // activation rows per MMA (a multiple of 32)
  int tmem_cols;
  int rows, stages;
  float* P;                 // PLAIN: P[split][row][feature]
  size_t split_stride;
  int ld;
  float* scratch;           // [pair][cta][quad of rows][128 features] float4: partial sums of a pair's first segment
  int* flags;               // [pair][cta]; zero between launches (whoever consumes a flag lowers it; a launch in which a wait gave up
                            // may leave one raised: whoever clears the error word clears them too)
  float* x;                 // RESID: residual rows, updated in place
  const __nv_bfloat16* gain;      // the next norm's gain, or NULL: x only
  __nv_bfloat16* xn;        // gain * x
  float* ss;                // [row][out / 128] sums of squares
  int out;
  __nv_bfloat16* act;       // SWIGLU
  int f, up_first;
  RowScale rs;
  __nv_bfloat16* q;         // ROPE
  RopeGroups gr;
  int n_heads, dh, max_ctx;
  int wait_first;           // see tc_gemm_wait_first
  int* err_flag;
  unsigned long long wait_limit_ns;
  uint32_t extra_tx;        // self-test only: bytes that a pair's first stage expects beyond what is copied
};

struct Segment { int tile, u0, u1; };     // units [u0, u1) of a tile's K range

// The segments of one group's range of work units, in order.
struct SegIter {
  int u, end, upt;
  __device__ bool next(Segment& s) {
    if (u >= end) return false;
    const int t = u / upt;
    s.tile = t;
    s.u0 = u - t * upt;
    s.u1 = end - t * upt < upt ? end - t * upt : upt;
    u = t * upt + s.u1;
    return true;
  }
};

// First work unit of a group; range_begin(group + 1) is its end.
__device__ __forceinline__ int range_begin(const WideParams& prm, int group) {
  if (prm.splits == 0) return prm.range[group];
  const int t = group / prm.splits, s = group - t * prm.splits;
  return t * prm.units_per_tile + s * prm.units_per_tile / prm.splits;
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
__device__ __forceinline__ uint32_t cluster_id() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Execution order only (see the uses).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); }
// shared memory of this CTA -> shared memory of a CTA of the cluster; the bytes are counted by a barrier there
__device__ __forceinline__ void bulk_to_peer(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "r"(smem_u32(src)), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ float4 bf16x4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u), __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
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
__device__ __forceinline__ void umma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
// Arrives at the same barrier of both CTAs once the MMAs issued so far are complete.
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar, uint32_t lead) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"((uint16_t)(3u << lead)) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\ttcgen05.wait::ld.sync.aligned;"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
#pragma unroll
  for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(r[e]);
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory"); }

// The fused forms combine two features of a tile that sit in different TMEM lanes (gate / up, or the members of a rotation
// pair), so a batch of rows goes through shared memory in fp32: warps park 32 features x 8 rows at a time, then every thread
// finishes four neighbouring outputs (pairs) of a row.  Combining them by shuffles between the lanes that hold them took three
// times the instructions (about 300 per warp and 16 rows).  A batch is 32 rows while the ring is in use; behind the pair's last
// main loop the ring is free and all rows are one batch, because each batch costs a round trip to the partial sums in L2 and
// two barriers (about 1 us): 256 rows in batches of 32 kept that last, exposed epilogue at 9-11 us.
constexpr int kChunk = 8;                               // activation rows a warp takes from tensor memory at a time
constexpr int kBatch = kEpiThreads / 128 * kChunk;      // rows of a batch
constexpr int kPark = kBatch * kTileM * 4;              // bytes

template <int EPI, int KB>
__global__ void __launch_bounds__(kWideThreads, 1)
tc_wide_kernel(const __grid_constant__ WideMaps maps, const WideParams prm) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr bool SCALED = EPI == WIDE_SWIGLU || EPI == WIDE_ROPE;   // the activation rows' RMS division is still to be done
  __shared__ float inv_s[SCALED ? 256 : 1];                        // 1 / rms of this pair's activation rows
  __shared__ __nv_bfloat16* dst_s[EPI == WIDE_ROPE ? 256 : 1];     // where the segment's matrix (q, k or v) of a row goes, NULL: nowhere
  __shared__ const float2* table_s[EPI == WIDE_ROPE ? 256 : 1];    // its rotary table row
  __shared__ __align__(8) uint64_t full_bar[kMaxStages], empty_bar[kMaxStages], accum_full[2], accum_empty[2], recv_full;
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;

  // The way to the first MMA is a chain of latencies of about a microsecond each, so they run side by side: every warp arrives
  // at the cluster's barrier as soon as its own part is done (barriers initialised, tensor memory allocated) and waits for it
  // only where it needs the others; warp 0 issues the weights while warp 1 waits for the kernel before this one and then fetches
  // the ring's first activations.  One after the other, it took 4.9 us from the CTA's start to the first full stage.
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < prm.stages; ++s) { mbar_init(&full_bar[s], 1); mbar_init(&empty_bar[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&accum_full[s], 1); mbar_init(&accum_empty[s], 2 * kEpiThreads / 32); }
    mbar_init(&recv_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)), "r"(prm.tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    pdl_launch_dependents();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncwarp();
  cluster_arrive_release();
  const uint32_t crank = cluster_rank(), rank = crank & 1u, lead = crank & ~1u;     // in the cluster, in the pair; the pair's even CTA
  int pair = prm.groups * prm.nrb - 1 - (int)(blockIdx.x >> 1);              // against the launch order (see above)
  int group = prm.nrb == 2 ? pair >> 1 : pair, rb = prm.nrb == 2 ? pair & 1 : 0;
  if constexpr (EPI == WIDE_RESID) {                                         // a cluster holds the splits of one tile and row block
    const int item = (int)cluster_id();
    rb = prm.nrb == 2 ? item & 1 : 0;
    group = (prm.nrb == 2 ? item >> 1 : item) * prm.splits + (int)(crank >> 1);
  }
  const int stages = prm.stages, n = prm.n;
  const uint32_t b_tile = (uint32_t)n / 2 * 128, a_tile = kTileM * 128;         // one K block of each operand
  const uint32_t stage_bytes = KB * (a_tile + b_tile);
  const unsigned long long limit_ns = prm.wait_limit_ns;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float* const small_park = reinterpret_cast<float*>(smem + (size_t)stages * stage_bytes); // fused forms: [kBatch][128]
  const SegIter first = {range_begin(prm, group), range_begin(prm, group + 1), prm.units_per_tile};
  auto load_x = [&](int st, int u) {
    const uint32_t bar = map_to_rank(smem_u32(&full_bar[st]), lead);
    tma_pair_3d(smem + (size_t)st * stage_bytes + KB * a_tile, &maps.x, 0, rb * n + (int)rank * (n / 2), u * KB, bar);
  };
  // both CTAs' barriers and tensor memory exist behind this
  auto cluster_ready = [&]() {
    cluster_wait_acquire();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };

  if (warp == 0) {
    // ---------------- TMA producer of this CTA's half of the operands
    const bool leader = elect_one();
    const uint64_t wpol = l2_evict_first_policy();
    // a division by a run-time value is about 170 clocks, so a segment's matrix and tile are worked out once, and ring position and
    // parity are counted
    int seg = 0, lt = 0;
    auto next_segment = [&](SegIter& it, Segment& s) {
      const bool more = it.next(s);
      if (more) { seg = s.tile / prm.tiles_per_seg; lt = s.tile - seg * prm.tiles_per_seg; }
      return more;
    };
    auto load_w = [&](int st, int u, uint32_t more) {
      const uint32_t bar = map_to_rank(smem_u32(&full_bar[st]), lead);
      uint8_t* dst = smem + (size_t)st * stage_bytes;
      if (rank == 0) mbar_expect_tx(&full_bar[st], 2 * stage_bytes + more);
      if (EPI == WIDE_SWIGLU) tma_pair_4d(dst, &maps.w[0], 0, (lt * 2 + (int)rank) * (kTileM / 2), 0, u * KB, bar, wpol);
      else tma_pair_3d(dst, &maps.w[seg], 0, (lt * 2 + (int)rank) * kTileM, u * KB, bar, wpol);
    };
    // weights do not depend on the kernel before: fill the ring with them; warp 1 fetches those stages' activations
    if (prm.wait_first) pdl_wait();
    cluster_ready();
    SegIter it = first;
    Segment sg;
    bool have = next_segment(it, sg);
    int u = have ? sg.u0 : 0, i = 0;
    for (; i < stages && have; ++i) {
      if (leader) load_w(i, u, i == 0 ? prm.extra_tx : 0u);
      if (++u == sg.u1) { have = next_segment(it, sg); u = sg.u0; }
    }
    __syncwarp();
    pdl_wait();
    for (int st = 0, ph = 0; have; ++i) {
      if (!__all_sync(0xffffffffu, mbar_wait(&empty_bar[st], ph, &abort_flag, limit_ns))) break;
      if (leader) { load_w(st, u, 0u); load_x(st, u); }
      __syncwarp();
      if (++u == sg.u1) { have = next_segment(it, sg); u = sg.u0; }
      if (++st == stages) { st = 0; ph ^= 1; }
    }
    for (int j = i > stages ? i - stages : 0; j < i; ++j)  // every commit to this CTA's barriers has arrived
      if (!__all_sync(0xffffffffu, mbar_wait(&empty_bar[j % stages], (j / stages) & 1, &abort_flag, limit_ns))) break;
    if (abort_flag && rank == 0 && lane == 0) {          // drain: both CTAs' copies signal the even CTA's barriers
      for (int j = i > stages ? i - stages : 0; j < i; ++j) {
        const unsigned long long t0 = now_ns();
        while (!mbar_try(&full_bar[j % stages], (j / stages) & 1) && now_ns() - t0 < kDrainNs) {}
      }
    }
  } else if (warp == 1) {
    // ---------------- the ring's first activations, then MMA issuer (even CTA)
    const bool leader = elect_one();
    pdl_wait();
    cluster_ready();
    {
      SegIter it = first;
      Segment sg;
      bool have = it.next(sg);
      int u = have ? sg.u0 : 0;
      for (int i = 0; i < stages && have; ++i) {
        if (leader) load_x(i, u);
        if (++u == sg.u1) { have = it.next(sg); u = sg.u0; }
      }
      __syncwarp();
    }
    if (rank == 0) {
      const uint32_t tmem_d = tmem_base_slot;
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);
      SegIter it = first;
      Segment sg;
      bool ok = true;
      int st = 0, ph = 0;
      for (int j = 0; ok && it.next(sg); ++j) {
        const int as = j & 1, around = j >> 1;
        if (around > 0) ok = __all_sync(0xffffffffu, mbar_wait(&accum_empty[as], (around & 1) ^ 1, &abort_flag, limit_ns));
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d = tmem_d + (uint32_t)(as * n);
        for (int u = sg.u0; ok && u < sg.u1; ++u) {
          ok = __all_sync(0xffffffffu, mbar_wait(&full_bar[st], ph, &abort_flag, limit_ns));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (leader) {                                  // K blocks past the end of K have arrived as zeros
            const uint32_t a_addr = smem_u32(smem + (size_t)st * stage_bytes);
#pragma unroll
            for (int kk = 0; kk < KB; ++kk) {
              const uint64_t ad = umma_desc(a_addr + kk * a_tile), bd = umma_desc(a_addr + KB * a_tile + kk * b_tile);
#pragma unroll
              for (int k = 0; k < kTileK / kUmmaK; ++k)
                umma_pair(d, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), idesc, u > sg.u0 || kk > 0 || k > 0 ? 1u : 0u);
            }
            umma_commit_pair(&empty_bar[st], lead);
          }
          __syncwarp();
          if (++st == stages) { st = 0; ph ^= 1; }
        }
        if (ok && leader) umma_commit_pair(&accum_full[as], lead);
        __syncwarp();
      }
    }
  } else {
    // ---------------- epilogue
    const int quarter = warp & 3, sub = (warp - 2) >> 2, et = threadIdx.x - 64;
    const int row0 = rb * n, my_rows = prm.rows - row0 < n ? prm.rows - row0 : n;
    cluster_ready();
    const uint32_t tmem_d = tmem_base_slot;
    pdl_wait();
    if constexpr (SCALED) {
      if (et < my_rows) inv_s[et] = row_scale(prm.rs, row0 + et);
    }
    int my_group = 0, my_slot = -1;                      // ROPE: of row et
    if constexpr (EPI == WIDE_ROPE) {
      if (et < my_rows) {
        my_group = (row0 + et) / prm.gr.rpg;
        const int rl = row0 + et - my_group * prm.gr.rpg;
        const RowMeta* meta = prm.gr.meta[my_group];
        const int slot = meta->slot[rl];
        my_slot = rl < meta->n_rows && slot >= 0 && slot < prm.max_ctx ? slot : -1;
        table_s[et] = prm.gr.rope[my_group] + (size_t)rl * (prm.dh >> 1);
      }
    }
    epi_sync();
    const size_t slot_quads = (size_t)(n / 4) * kTileM;  // float4s of one CTA's partial sums
    const int frow = quarter * 32 + lane;                // row of this CTA's tile
    float4* const scratch = reinterpret_cast<float4*>(prm.scratch) + frow;
    SegIter it = first;
    Segment sg;
    bool left = false;
    auto leave = [&]() {                                 // nothing more of this warp's concerns the partner
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (EPI == WIDE_RESID) cluster_arrive();
      else cluster_arrive_release();                     // behind the arrivals at the partner's barrier
      left = true;
    };
    for (int j = 0; it.next(sg); ++j) {
      const bool last = it.u >= it.end;                  // the ring is free, nothing waits for the accumulator
      const int as = j & 1;
      // RESID: rows [lo, hi) are this CTA's share, a warp finishes whole rows of the tile's 128 features, four features a lane;
      // the old values are fetched while the main loop runs
      constexpr int kAhead = 8, kRowWarps = kEpiThreads / 32;
      const int S = prm.splits, split = (int)(crank >> 1), per = EPI == WIDE_RESID ? ((n + S - 1) / S + 7) / 8 * 8 : 0;
      const int lo = split * per, hi = lo + per < my_rows ? lo + per : my_rows, f0 = sg.tile * 256 + (int)rank * kTileM + lane * 4;
      float4 old[kAhead], gn;
      auto fetch_old = [&](int r) {
#pragma unroll
        for (int q = 0; q < kAhead; ++q)
          if (r + q * kRowWarps < hi) old[q] = *reinterpret_cast<const float4*>(prm.x + (size_t)(row0 + r + q * kRowWarps) * prm.out + f0);
      };
      if constexpr (EPI == WIDE_RESID) {
        if (prm.gain != nullptr) gn = bf16x4(prm.gain + f0);
        fetch_old(lo + (et >> 5));
      }
      bool ok = __all_sync(0xffffffffu, mbar_wait(&accum_full[as], (j >> 1) & 1, &abort_flag, limit_ns));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t t0 = tmem_d + (uint32_t)(as * n) + ((uint32_t)(quarter * 32) << 16);
      auto release = [&]() {                             // this warp has read the accumulator
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_u32(&accum_empty[as]), lead));
      };
      if constexpr (EPI == WIDE_RESID) {
        float* const park = reinterpret_cast<float*>(smem);                    // [n][128]: the ring is free
        uint8_t* const recv = smem + (size_t)n * kTileM * 4;                   // the other splits' sums of this CTA's share
        const uint32_t share = (uint32_t)per * kTileM * 4;
        __syncwarp();
        cluster_arrive();                                 // this CTA's MMAs have read their operands: peers may write here
        // The shares go out one by one while the next is read from tensor memory, this CTA's own comes last.  A warp reads
        // pieces of 8 rows; a share begins where a piece does.
        for (int i = 1; i <= S; ++i) {
          const int o = split + i < S ? split + i : split + i - S, olo = o * per, ohi = olo + per < my_rows ? olo + per : my_rows;
          for (int r = olo + sub * kChunk; r < ohi; r += kBatch) {
            float v[kChunk];
            tmem_ld8(t0 + (uint32_t)r, v);
#pragma unroll
            for (int e = 0; e < kChunk; ++e) park[(r + e) * kTileM + frow] = ok ? v[e] : 0.f;
          }
          if (i < S) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the copies read through the async proxy
          epi_sync();
          if (i == 1) { __syncwarp(); cluster_wait(); }
          if (i < S && et == 0 && ohi > olo) {
            const uint32_t to = (uint32_t)o * 2 + rank;
            bulk_to_peer(map_to_rank(smem_u32(recv + (size_t)(split < o ? split : split - 1) * share), to), park + (size_t)olo * kTileM,
                         (uint32_t)(ohi - olo) * kTileM * 4, map_to_rank(smem_u32(&recv_full), to));
          }
          __syncwarp();
        }
        if (et == 0) mbar_expect_tx(&recv_full, hi > lo ? (uint32_t)(S - 1) * (uint32_t)(hi - lo) * kTileM * 4 : 0u);
        __all_sync(0xffffffffu, mbar_wait(&recv_full, 0, &abort_flag, limit_ns));
        leave();
        for (int rl = lo + (et >> 5); rl < hi; rl += kAhead * kRowWarps) {
          if (rl != lo + (et >> 5)) fetch_old(rl);
#pragma unroll
          for (int q = 0; q < kAhead; ++q) {
            const int r = rl + q * kRowWarps;
            if (r >= hi) continue;                        // uniform over the warp
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int s = 0; s < S; ++s) {                 // in K order
              const float4 p = s == split ? *reinterpret_cast<const float4*>(park + (size_t)r * kTileM + lane * 4)
                                          : *reinterpret_cast<const float4*>(recv + (size_t)(s < split ? s : s - 1) * share + ((size_t)(r - lo) * kTileM + lane * 4) * 4);
              a.x += p.x; a.y += p.y; a.z += p.z; a.w += p.w;
            }
            float4 v = old[q];
            v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
            *reinterpret_cast<float4*>(prm.x + (size_t)(row0 + r) * prm.out + f0) = v;
            if (prm.gain == nullptr) continue;
            const __nv_bfloat162 y0 = __floats2bfloat162_rn(gn.x * v.x, gn.y * v.y), y1 = __floats2bfloat162_rn(gn.z * v.z, gn.w * v.w);
            *reinterpret_cast<uint2*>(prm.xn + (size_t)(row0 + r) * prm.out + f0) =
                make_uint2(*reinterpret_cast<const uint32_t*>(&y0), *reinterpret_cast<const uint32_t*>(&y1));
            float sq = v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
            for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
            if (lane == 0) prm.ss[(size_t)(row0 + r) * (prm.out / kTileM) + sg.tile * 2 + rank] = sq;
          }
        }
        continue;
      }
      if (prm.splits == 0 && sg.u0 > 0) {                // not the tile's first K columns: leave the sums to the pair that has them
        float4* dst = scratch + ((size_t)pair * 2 + rank) * slot_quads;
        for (int r = sub * kChunk; ok && r < my_rows; r += kBatch) {
          float v[kChunk];
          tmem_ld8(t0 + (uint32_t)r, v);
          __stcg(dst + (size_t)(r / 4) * kTileM, make_float4(v[0], v[1], v[2], v[3]));
          __stcg(dst + (size_t)(r / 4 + 1) * kTileM, make_float4(v[4], v[5], v[6], v[7]));
        }
        if (last) leave();
        else release();
        __threadfence();
        epi_sync();
        if (et == 0) asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(prm.flags + pair * 2 + rank), "r"(1) : "memory");
        continue;
      }
      int helpers = 0;                                    // groups after this one that hold the rest of the tile
      if (prm.splits == 0 && sg.u1 < prm.units_per_tile) {
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
        ok = __all_sync(0xffffffffu, ok && *(volatile int*)&abort_flag == 0);
      }
      // a wait that gave up: the plain form writes nothing.  Uniform over the epilogue warps only behind a barrier, so the fused forms,
      // which need barriers of their own, run through with whatever the accumulator holds; the end of the kernel replaces both.
      const int seg = sg.tile / prm.tiles_per_seg, lt = sg.tile - seg * prm.tiles_per_seg;
      const float4* src = scratch + ((size_t)(pair + prm.nrb) * 2 + rank) * slot_quads;
      const size_t next_helper = (size_t)prm.nrb * 2 * slot_quads;
      // Sums of rows r .. r + 7 over all K; the partial sums' loads are in flight before the first use.
      auto load_rows = [&](int r, float* v) {
        float4 o0, o1;
        const float4* p = src + (size_t)(r / 4) * kTileM;
        if (helpers > 0) { o0 = __ldcg(p); o1 = __ldcg(p + kTileM); }
        tmem_ld8(t0 + (uint32_t)r, v);
        for (int hp = 0; hp < helpers; ++hp) {
          v[0] += o0.x; v[1] += o0.y; v[2] += o0.z; v[3] += o0.w;
          v[4] += o1.x; v[5] += o1.y; v[6] += o1.z; v[7] += o1.w;
          if (hp + 1 < helpers) {
            p += next_helper;
            o0 = __ldcg(p);
            o1 = __ldcg(p + kTileM);
          }
        }
      };
      if constexpr (EPI == WIDE_PLAIN) {
        const int split = prm.splits > 0 ? group % prm.splits : 0;
        float* out = prm.P + (size_t)split * prm.split_stride + (size_t)(row0 + sub * kChunk) * prm.ld + (size_t)sg.tile * 256 + rank * kTileM + frow;
        for (int r = sub * kChunk; ok && r < my_rows; r += kBatch, out += (size_t)kBatch * prm.ld) {
          float v[kChunk];
          load_rows(r, v);
#pragma unroll
          for (int e = 0; e < kChunk; ++e)
            if (r + e < my_rows) out[(size_t)e * prm.ld] = v[e];
        }
        if (!last) release();
      } else {
        // item i of a batch: row i / 16, outputs 4 (i % 16) .. + 3 (SwiGLU) or as many rotation pairs
        const int p4 = (et & 15) * 4;
        const int hdim = prm.dh >> 1;
        // SwiGLU: lo = gate, hi = up, in the order they have in the tile
        const int lo_at = EPI == WIDE_ROPE ? p4 / hdim * prm.dh + p4 % hdim : prm.up_first ? p4 + kTileM / 2 : p4;
        const int hi_at = EPI == WIDE_ROPE ? lo_at + hdim : prm.up_first ? p4 : p4 + kTileM / 2;
        const int head = EPI == WIDE_ROPE ? (lt * 2 + (int)rank) * kTileM / prm.dh + p4 / hdim : 0;
        // what a row's address needs is worked out once per segment and row, not per row and thread
        const size_t col = EPI == WIDE_ROPE ? (size_t)head * (seg == 0 ? prm.dh : prm.max_ctx * prm.dh) + p4 % hdim
                                            : (size_t)(lt * 2 + (int)rank) * (kTileM / 2) + p4;
        if constexpr (EPI == WIDE_ROPE) {
          if (et < my_rows)
            dst_s[et] = seg == 0 ? prm.q + (size_t)(row0 + et) * prm.n_heads * prm.dh
                                 : my_slot < 0 ? nullptr : (__nv_bfloat16*)(seg == 1 ? prm.gr.kc[my_group] : prm.gr.vc[my_group]) + (size_t)my_slot * prm.dh;
        }
        float* const park = last ? reinterpret_cast<float*>(smem) : small_park;
        const int batch = last ? my_rows : kBatch;
        for (int b0 = 0; b0 < my_rows; b0 += batch) {
          const int b1 = b0 + batch < my_rows ? b0 + batch : my_rows;
#pragma unroll 2
          for (int r = b0 + sub * kChunk; r < b1; r += kBatch) {
            float v[kChunk];
            load_rows(r, v);
#pragma unroll
            for (int e = 0; e < kChunk; ++e) park[(r - b0 + e) * kTileM + frow] = v[e];
          }
          if (b1 == my_rows) {
            if (last) leave();
            else release();
          }
          epi_sync();
#pragma unroll 2
          for (int rl = b0 + (et >> 4); rl < b1; rl += kEpiThreads / 16) {
            const float sc = inv_s[rl];
            float4 cs0 = make_float4(1.f, 0.f, 1.f, 0.f), cs1 = cs0;
            if (EPI == WIDE_ROPE && seg < 2) {
              const float4* t = reinterpret_cast<const float4*>(table_s[rl] + p4 % hdim);
              cs0 = __ldg(t);
              cs1 = __ldg(t + 1);
            }
            const float* row = park + (rl - b0) * kTileM;
            float4 a = *reinterpret_cast<const float4*>(row + lo_at), b = *reinterpret_cast<const float4*>(row + hi_at);
            a.x *= sc; a.y *= sc; a.z *= sc; a.w *= sc; b.x *= sc; b.y *= sc; b.z *= sc; b.w *= sc;
            if constexpr (EPI == WIDE_SWIGLU) {
              const __nv_bfloat162 y0 = __floats2bfloat162_rn(__fdividef(a.x, 1.0f + __expf(-a.x)) * b.x, __fdividef(a.y, 1.0f + __expf(-a.y)) * b.y);
              const __nv_bfloat162 y1 = __floats2bfloat162_rn(__fdividef(a.z, 1.0f + __expf(-a.z)) * b.z, __fdividef(a.w, 1.0f + __expf(-a.w)) * b.w);
              *reinterpret_cast<uint2*>(prm.act + (size_t)(row0 + rl) * prm.f + col) =
                  make_uint2(*reinterpret_cast<const uint32_t*>(&y0), *reinterpret_cast<const uint32_t*>(&y1));
            } else {
              __nv_bfloat16* const row_dst = dst_s[rl];
              if (row_dst != nullptr) {
                __nv_bfloat16* const dst = row_dst + col;
                const __nv_bfloat162 l0 = __floats2bfloat162_rn(a.x * cs0.x - b.x * cs0.y, a.y * cs0.z - b.y * cs0.w);
                const __nv_bfloat162 l1 = __floats2bfloat162_rn(a.z * cs1.x - b.z * cs1.y, a.w * cs1.z - b.w * cs1.w);
                const __nv_bfloat162 h0 = __floats2bfloat162_rn(b.x * cs0.x + a.x * cs0.y, b.y * cs0.z + a.y * cs0.w);
                const __nv_bfloat162 h1 = __floats2bfloat162_rn(b.z * cs1.x + a.z * cs1.y, b.w * cs1.z + a.w * cs1.w);
                *reinterpret_cast<uint2*>(dst) = make_uint2(*reinterpret_cast<const uint32_t*>(&l0), *reinterpret_cast<const uint32_t*>(&l1));
                *reinterpret_cast<uint2*>(dst + hdim) = make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
              }
            }
          }
          if (!last) epi_sync();                          // the batch's rows have been read
        }
      }
      if (helpers > 0) {                                  // every thread has read the sums: lower the flags for the next launch
        if (EPI == WIDE_PLAIN) epi_sync();
        if (et < helpers) prm.flags[(pair + (1 + et) * prm.nrb) * 2 + rank] = 0;
      }
    }
    if (!left) leave();
  }
  // No CTA leaves, and no tensor memory is given back, while the partner may still signal, read or write this CTA's memory: all
  // warps arrive at the cluster's barrier behind their last such step, which for the epilogue is well before its last stores, so
  // the wait costs nothing (with all arrivals at the very end the 128-node tree's step loop took 25.45 ms, now 25.28).
  if (warp < 2) {
    __syncwarp();
    cluster_arrive();
    if (EPI == WIDE_RESID) {                              // (the epilogue's first barrier)
      cluster_wait();
      cluster_arrive();
    }
  }
  cluster_wait();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base_slot), "r"(prm.tmem_cols) : "memory");
  }
  __syncthreads();
  if (abort_flag) {
    // A wait gave up.  Zeros in place of whatever this CTA has written: the caches must hold finite values whatever happens, because
    // attention fetches whole tiles of them and masks by a probability of zero.  Out of the way of the main path: a test per batch
    // of the epilogue cost a prefill of 128 tokens 0.4 %.
    SegIter it = {range_begin(prm, group), range_begin(prm, group + 1), prm.units_per_tile};
    Segment sg;
    const int row0 = rb * n, my_rows = prm.rows - row0 < n ? prm.rows - row0 : n;
    const __nv_bfloat16 zero = __float2bfloat16(0.f);
    while (it.next(sg)) {
      if (prm.splits == 0 && sg.u0 > 0) continue;          // the pair that has the tile's first K columns writes it
      const int seg = sg.tile / prm.tiles_per_seg, lt = sg.tile - seg * prm.tiles_per_seg;
      for (int i = threadIdx.x; i < my_rows * kTileM; i += kWideThreads) {
        const int r = i / kTileM, c = i - r * kTileM, row = row0 + r;
        if constexpr (EPI == WIDE_PLAIN) {
          prm.P[(size_t)(prm.splits > 0 ? group % prm.splits : 0) * prm.split_stride + (size_t)row * prm.ld + (size_t)sg.tile * 256 + rank * kTileM + c] = 0.f;
        } else if constexpr (EPI == WIDE_SWIGLU) {
          if (c < kTileM / 2) prm.act[(size_t)row * prm.f + (size_t)(lt * 2 + (int)rank) * (kTileM / 2) + c] = zero;
        } else if constexpr (EPI == WIDE_ROPE) {
          const int g = row / prm.gr.rpg, rl = row - g * prm.gr.rpg, feat = (lt * 2 + (int)rank) * kTileM + c, head = feat / prm.dh;
          const RowMeta* meta = prm.gr.meta[g];
          const int slot = meta->slot[rl];
          if (seg == 0) prm.q[(size_t)row * prm.n_heads * prm.dh + feat] = zero;
          else if (rl < meta->n_rows && slot >= 0 && slot < prm.max_ctx)
            ((__nv_bfloat16*)(seg == 1 ? prm.gr.kc[g] : prm.gr.vc[g]))[((size_t)head * prm.max_ctx + slot) * prm.dh + feat - head * prm.dh] = zero;
        } else {
          const int per = ((n + prm.splits - 1) / prm.splits + 7) / 8 * 8, lo = (int)(crank >> 1) * per;      // this CTA's share of the rows
          if (r < lo || r >= lo + per) continue;
          const size_t at = (size_t)row * prm.out + (size_t)sg.tile * 256 + rank * kTileM + c;
          prm.x[at] = 0.f;
          if (prm.gain != nullptr) prm.xn[at] = zero;
          if (prm.gain != nullptr && c == 0) prm.ss[(size_t)row * (prm.out / kTileM) + sg.tile * 2 + rank] = 0.f;
        }
      }
    }
    if (threadIdx.x == 0 && prm.err_flag) *prm.err_flag = AMPH_ERR_TIMEOUT;
  }
}

constexpr size_t kWideSmem = 220 * 1024;                  // ring + alignment; the static part needs up to 6 KB of the 227
constexpr size_t kResidSmem = 225 * 1024;                 // 256 parked rows and three quarters of them received; 1 KB static

// Clusters of `ctas` that run at a time (0: none, or the question failed).
int active_clusters(const TcGemm* g, const void* kernel, int ctas, size_t smem) {
  int n = 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g->sm_count / ctas * ctas);
  cfg.blockDim = dim3(kWideThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
  return n;
}
template <int EPI>
constexpr size_t ring_smem() { return EPI == WIDE_RESID ? kResidSmem : kWideSmem; }
// Raises the shared memory limit of a form that is about to be launched, once per plan set: amph_project makes one per call, and three forms
// more than it needs cost it 0.5 us (100 rows: 10.5 us of host time, now 9.9).
template <int EPI, int KB>
bool allow_smem(TcGemm* g) {
  bool& ready = g->wide_ready[EPI][KB - 1];
  if (!ready) ready = cudaFuncSetAttribute(tc_wide_kernel<EPI, KB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ring_smem<EPI>()) == cudaSuccess;
  if (!ready) cudaGetLastError();
  return ready;
}
// K blocks of a stage.  One, so that six are in flight, where a block's MMAs take longer than the step from one stage to the next (two
// barrier waits, a commit, two copies) and K is long: 4 x 64 rows at 4096, 8 layers, 12 steps 28.4 ms with two (three stages), 27.9 with
// one, a prompt of 300 tokens 1970 / 1910 us.  Two otherwise: trees of 70 / 96 / 128 nodes at 4096 with one block 8150 / 8230 / 8500 us
// (8 layers, 6 steps), with two 7990 / 8090 / 8370, a prompt of 100 tokens 1400 / 1375; 8 x 64 rows at width 512 495 / 487 us a step, at
// 1024 607 / 597, at 2048 (K = 5632 in the down projection) 801 / 805.
int unit_kb(int in, int rows) { return rows <= 128 || in <= 2816 ? 2 : 1; }

// What runs at a time, asked for by the first launch that may take the kernel (or by tc_wide_init): amph_project makes a plan set
// per call, mostly for fewer rows, and needs the plain form only (16 rows: 14.7 us of host time per call when every plan set asked for
// everything, 13.5 now; 100 rows 10.8, now 9.7).
bool wide_available(TcGemm* g) {
  if (!g) return false;
  if (g->wide_pairs < 0) {
    g->wide_pairs = 0;
    if ((size_t)g->max_smem >= kWideSmem + 7 * 1024 && allow_smem<WIDE_ROPE, 1>(g)) {
      const int clusters = active_clusters(g, (const void*)tc_wide_kernel<WIDE_ROPE, 1>, 2, kWideSmem);
      g->wide_pairs = clusters < g->sm_count / 2 ? clusters : g->sm_count / 2;
    }
  }
  return g->wide_pairs > 1;
}
// clusters of 1 .. 4 pairs of the residual form
bool resid_available(TcGemm* g) {
  if (!wide_available(g)) return false;
  if (g->resid_clusters[0] == 0) {
    g->resid_clusters[0] = 1;
    if (allow_smem<WIDE_RESID, 1>(g))
      for (int s = 1; s <= 4; ++s) g->resid_clusters[s] = active_clusters(g, (const void*)tc_wide_kernel<WIDE_RESID, 1>, 2 * s, kResidSmem);
  }
  return true;
}

// Everything of a launch that does not depend on the epilogue; false: the shape is not covered.
template <int EPI>
bool wide_params(TcGemm* g, int xb, int n_seg, int tiles_per_seg, int in, int rows, int splits, float* scratch_end, size_t scratch_floats,
                 WideMaps* maps, WideParams* prm) {
  constexpr size_t out_bytes = EPI == WIDE_SWIGLU || EPI == WIDE_ROPE ? kPark : 0;
  if (!wide_available(g) || xb < 0 || xb >= g->n_x || g->xcols[xb] != in) return false;
  if (in % kTileK || rows < 32 || rows > kMaxWideRows || rows > g->xrows[xb] || n_seg < 1 || n_seg > kMaxSeg) return false;
  memset(maps, 0, sizeof *maps);
  memset(prm, 0, sizeof *prm);
  prm->nrb = rows > 256 ? 2 : 1;
  prm->n = ((rows + prm->nrb - 1) / prm->nrb + 31) / 32 * 32;        // an M = 256 pair MMA takes N in steps of 32
  const int kb = prm->kb = unit_kb(in, rows);
  const CUtensorMap* mx = g->get(g->xptr[xb], g->xrows[xb], in, prm->n / 2, kb);
  if (!mx) return false;
  maps->x = *mx;
  prm->tmem_cols = 64;
  while (prm->tmem_cols < 2 * prm->n) prm->tmem_cols *= 2;
  prm->tiles_per_seg = tiles_per_seg;
  prm->tiles = n_seg * tiles_per_seg;
  prm->kblocks = in / kTileK;
  prm->units_per_tile = (prm->kblocks + kb - 1) / kb;
  prm->splits = splits;
  prm->groups = g->wide_pairs / prm->nrb;
  const int units = prm->tiles * prm->units_per_tile;
  if (splits > 0) {
    if (splits > prm->units_per_tile) return false;
    prm->groups = prm->tiles * splits;
  } else {
    // at least 512 columns a group, unless there are more tiles than that; no more pairs than scratch
    const int most = units * kb / 8 > prm->tiles ? units * kb / 8 : prm->tiles;
    if (prm->groups > most) prm->groups = most;
    const size_t per_group = (size_t)prm->nrb * 2 * prm->n * kTileM;
    if ((size_t)prm->groups > scratch_floats / per_group) prm->groups = (int)(scratch_floats / per_group);
    if (prm->groups < 1 || !scratch_end || !g->wide_flags || 2 * prm->groups * prm->nrb > kWideFlags) return false;
    // a cut within `snap` units of a tile's edge moves to the edge: the piece it would leave costs a whole epilogue (5-10 us
    // when nothing runs above it) for a few K blocks of 0.3 us
    const int upt = prm->units_per_tile, share = units / prm->groups / 4, snap = share < upt / 8 ? share : upt / 8;
    for (int i = 0; i <= prm->groups; ++i) {
      int u = (int)((long long)i * units / prm->groups);
      const int rem = u % upt;
      if (rem <= snap) u -= rem;
      else if (rem >= upt - snap) u += upt - rem;
      prm->range[i] = u;
    }
    prm->scratch = scratch_end - (size_t)prm->groups * per_group;    // the buffer's end: its beginning may hold the result
  }
  prm->rows = rows;
  const size_t stage = kb * ((size_t)kTileM * 128 + (size_t)prm->n / 2 * 128);
  prm->stages = (int)((ring_smem<EPI>() - 1024 - out_bytes) / stage);
  if (prm->stages > kMaxStages) prm->stages = kMaxStages;
  prm->flags = g->wide_flags;
  prm->wait_first = g->wait_first;
  prm->err_flag = g->err_flag;
  prm->wait_limit_ns = g->wait_limit_ns;
  prm->extra_tx = g->extra_tx;
  return true;
}

template <int EPI>
bool wide_run(TcGemm* g, const WideMaps& maps, const WideParams& prm, cudaStream_t st) {
  if (!(prm.kb == 2 ? allow_smem<EPI, 2>(g) : allow_smem<EPI, 1>(g))) return false;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * prm.groups * prm.nrb);
  cfg.blockDim = dim3(kWideThreads);
  cfg.dynamicSmemBytes = ring_smem<EPI>();
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = EPI == WIDE_RESID ? 2 * prm.splits : 2;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, prm.kb == 2 ? tc_wide_kernel<EPI, 2> : tc_wide_kernel<EPI, 1>, maps, prm) == cudaSuccess;
}

}  // namespace

void tc_wide_init(TcGemm* g) { resid_available(g); }

void tc_wide_off(TcGemm* g) {
  g->wide_pairs = 0;
}

void tc_wide_bind(TcGemm* g, float* scratch, size_t scratch_floats, int* flags) {
  g->wide_scratch = scratch;
  g->wide_scratch_floats = scratch_floats / 64 * 64;
  g->wide_flags = flags;
}

bool tc_wide_launch(TcGemm* g, int xb, const void* const* w, int n_seg, int out, int in, int rows, float* P, size_t p_floats,
                    int* splits_out, size_t* split_stride, cudaStream_t st) {
  if (out % 256 || in % kTileK || !wide_available(g)) return false;
  const int tiles = n_seg * (out / 256);
  const size_t ld = (size_t)n_seg * out, stride = (size_t)rows * ld;
  if (stride > p_floats) return false;
  // Few tiles: the consumer adds the K ranges' sums (one per group).  Many: equal ranges of all the work, one sum.
  int splits = 0;
  const int groups = g->wide_pairs / (rows > 256 ? 2 : 1);
  if (tiles * 2 <= groups || !g->wide_flags) {
    splits = groups / tiles;
    if (splits > in / kTileK / 4) splits = in / kTileK / 4;            // at least four K blocks per pair
    if (splits > 16) splits = 16;
    while (splits > 1 && splits * stride > p_floats) --splits;
    if (splits < 1) splits = 1;
  }
  WideMaps maps;
  WideParams prm;
  // a cut tile's sums go to the end of the caller's buffer, behind the result
  const size_t end = p_floats / 64 * 64, used = (stride + 63) / 64 * 64;
  if (!wide_params<WIDE_PLAIN>(g, xb, n_seg, out / 256, in, rows, splits, P + end, end > used ? end - used : 0, &maps, &prm)) return false;
  for (int s = 0; s < n_seg; ++s) {
    if ((uintptr_t)w[s] & 15) return false;
    const CUtensorMap* m = g->get(w[s], out, in, kTileM, prm.kb);
    if (!m) return false;
    maps.w[s] = *m;
  }
  prm.P = P;
  prm.ld = (int)ld;
  prm.split_stride = stride;
  if (!wide_run<WIDE_PLAIN>(g, maps, prm, st)) return false;
  *splits_out = splits > 0 ? splits : 1;
  *split_stride = stride;
  return true;
}

bool tc_wide_launch_resid(TcGemm* g, int xb, const void* w, int out, int in, int rows, float* x, const void* gain, void* xn, float* ss,
                          cudaStream_t st) {
  if (!g || !w || !x || out % 256 || in % kTileK || ((uintptr_t)w & 15) || (gain && (!xn || !ss)) || !resid_available(g)) return false;
  // as many K ranges per tile as run at a time, at least four K blocks each
  const int items = out / 256 * (rows > 256 ? 2 : 1);
  int splits = 4;
  while (splits > 1 && (g->resid_clusters[splits] < items || splits > in / kTileK / 4)) --splits;
  if (g->resid_clusters[splits] < 1) return false;
  WideMaps maps;
  WideParams prm;
  if (!wide_params<WIDE_RESID>(g, xb, 1, out / 256, in, rows, splits, nullptr, 0, &maps, &prm)) return false;
  const CUtensorMap* m = g->get(w, out, in, kTileM, prm.kb);
  if (!m) return false;
  maps.w[0] = *m;
  prm.x = x;
  prm.gain = (const __nv_bfloat16*)gain;
  prm.xn = (__nv_bfloat16*)xn;
  prm.ss = ss;
  prm.out = out;
  return wide_run<WIDE_RESID>(g, maps, prm, st);
}

bool tc_wide_launch_swiglu(TcGemm* g, int xb, const void* w_gate, const void* w_up, int f, int in, int rows, void* act, const RowScale& rs,
                           cudaStream_t st) {
  if (!g || !g->wide_scratch || !w_gate || !w_up || !act || f % 128 || (((uintptr_t)w_gate | (uintptr_t)w_up) & 15)) return false;
  WideMaps maps;
  WideParams prm;
  if (!wide_params<WIDE_SWIGLU>(g, xb, 1, f / 128, in, rows, 0, g->wide_scratch + g->wide_scratch_floats, g->wide_scratch_floats, &maps, &prm)) return false;
  const bool up_first = (const char*)w_up < (const char*)w_gate;
  const uint64_t gap = up_first ? (const char*)w_gate - (const char*)w_up : (const char*)w_up - (const char*)w_gate;
  const CUtensorMap* m = g->get_halves(up_first ? w_up : w_gate, gap, f, in, kTileM / 2, prm.kb);
  if (!m) return false;
  maps.w[0] = *m;
  prm.act = (__nv_bfloat16*)act;
  prm.f = f;
  prm.up_first = up_first ? 1 : 0;
  prm.rs = rs;
  return wide_run<WIDE_SWIGLU>(g, maps, prm, st);
}

bool tc_wide_launch_qkv_rope(TcGemm* g, int xb, const void* wq, const void* wk, const void* wv, int n_heads, int dh, int in, int rows, void* q,
                             const RopeGroups& gr, int max_ctx, const RowScale& rs, cudaStream_t st) {
  const int d = n_heads * dh;
  if (!g || !g->wide_scratch || !wq || !wk || !wv || !q || (dh != 64 && dh != 128) || d % 256 || gr.rpg % 16) return false;
  if (((uintptr_t)wq | (uintptr_t)wk | (uintptr_t)wv) & 15) return false;
  WideMaps maps;
  WideParams prm;
  if (!wide_params<WIDE_ROPE>(g, xb, 3, d / 256, in, rows, 0, g->wide_scratch + g->wide_scratch_floats, g->wide_scratch_floats, &maps, &prm)) return false;
  const void* w[3] = {wq, wk, wv};
  for (int s = 0; s < 3; ++s) {
    const CUtensorMap* m = g->get(w[s], d, in, kTileM, prm.kb);
    if (!m) return false;
    maps.w[s] = *m;
  }
  prm.q = (__nv_bfloat16*)q;
  prm.gr = gr;
  prm.n_heads = n_heads;
  prm.dh = dh;
  prm.max_ctx = max_ctx;
  prm.rs = rs;
  return wide_run<WIDE_ROPE>(g, maps, prm, st);
}

}  // namespace amph
