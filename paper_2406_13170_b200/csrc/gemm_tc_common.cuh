// What the two tensor-core projection kernels share: barrier / TMA / descriptor helpers and the plan set (tensor maps).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <string.h>

#include <map>
#include <tuple>

#include "amph.h"
#include "amph_internal.cuh"
#include "gemm_tc.cuh"

namespace amph {
namespace tc {

constexpr int kTileM = 128;           // weight rows per CTA
constexpr int kTileK = 64;            // bf16 elements per 128-byte swizzle row
constexpr int kUmmaK = 16;            // K per tcgen05.mma for 16-bit inputs
constexpr int kStageKb = 2;           // 64-wide K blocks fetched by one TMA copy (one pipeline stage) when both operands' stage fits twice per CTA
constexpr int kMaxSeg = 8;
constexpr unsigned long long kWaitLimitNs = 1000000000ull;   // a barrier wait gives up after one second
constexpr unsigned long long kDrainNs = 10000000ull;         // what a CTA that gave up allows each of its copies to land (they take microseconds)

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait; returns false (and raises the shared abort flag) if the phase never completes or
// another role already gave up.
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag,
                                          unsigned long long limit_ns) {
  unsigned long long t0 = 0;
  for (uint32_t i = 1;; ++i) {
    if (mbar_try(bar, parity)) return true;
    if ((i & 63u) == 0u) {
      if (*abort_flag) return false;
      const unsigned long long t = now_ns();
      if (t0 == 0) t0 = t;
      else if (t - t0 > limit_ns) break;
    }
  }
  *abort_flag = 1;
  return false;
}

// One lane of a converged warp.  TMA and MMA instructions are issued by the elected lane while the other
// lanes stay with it: issued by a lone thread of a diverged warp, a tcgen05.mma costs about 210 clocks
// instead of the 48 that a 128 x 64 x 16 MMA occupies the tensor pipe (both measured), which would cap
// a CTA at about 37 GB/s of weights.
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0;
}

__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t umma_desc(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);          // start address
  d |= (uint64_t)1 << 16;                                // leading-dimension offset (unused with swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;                      // stride between 8-row groups
  d |= (uint64_t)1 << 46;                                // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                                // 128-byte swizzle
  return d;
}

typedef CUresult (*EncodeFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                             const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                             CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

}  // namespace tc

struct TcGemm {
  tc::EncodeFn encode = nullptr;
  int* err_flag = nullptr;
  int n_x = 0;
  void* xptr[16];
  int xrows[16], xcols[16];
  std::map<std::tuple<const void*, int, int, int, int>, CUtensorMap> cache;   // (ptr, rows, cols, box rows, box K blocks)
  int sm_count = 148;
  int max_smem = 0;
  unsigned long long wait_limit_ns = tc::kWaitLimitNs;
  uint32_t extra_tx = 0;
  int wait_first = 0;
  std::map<std::tuple<const void*, const void*, int, int, int>, CUtensorMap> pair_cache;   // (lower, upper matrix, rows, cols, K blocks)

  // Two [rows, cols] matrices as one 4-D tensor (column, row, K block, matrix): a box of 64 rows of both.
  const CUtensorMap* get_pair(const void* lo, const void* hi, int rows, int cols, int box_kb) {
    auto key = std::make_tuple(lo, hi, rows, cols, box_kb);
    auto it = pair_cache.find(key);
    if (it != pair_cache.end()) return &it->second;
    const uint64_t gap = (uint64_t)((const char*)hi - (const char*)lo);
    if (gap == 0 || (gap & 15) || gap >= (1ull << 40)) return nullptr;
    CUtensorMap m;
    const cuuint64_t dims[4] = {(cuuint64_t)tc::kTileK, (cuuint64_t)rows, (cuuint64_t)cols / tc::kTileK, 2};
    const cuuint64_t strides[3] = {(cuuint64_t)cols * 2, (cuuint64_t)tc::kTileK * 2, (cuuint64_t)gap};
    const cuuint32_t box[4] = {(cuuint32_t)tc::kTileK, (cuuint32_t)(tc::kTileM / 2), (cuuint32_t)box_kb, 2};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(lo), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return nullptr;
    return &(pair_cache[key] = m);
  }

  // Rows [0, rows) of a matrix and the rows `gap` bytes behind them, as (column, row, half, K block): a box is box_rows rows of
  // both halves per K block, one after the other.  The halves are two matrices, or the two halves of a head's rotation pairs (which
  // makes the tensor's last rows end behind the matrix: no box asks for those).
  std::map<std::tuple<const void*, uint64_t, int, int, int, int>, CUtensorMap> halves_cache;
  const CUtensorMap* get_halves(const void* ptr, uint64_t gap, int rows, int cols, int box_rows, int box_kb) {
    auto key = std::make_tuple(ptr, gap, rows, cols, box_rows, box_kb);
    auto it = halves_cache.find(key);
    if (it != halves_cache.end()) return &it->second;
    if (gap == 0 || (gap & 15) || gap >= (1ull << 40)) return nullptr;
    CUtensorMap m;
    const cuuint64_t dims[4] = {(cuuint64_t)tc::kTileK, (cuuint64_t)rows, 2, (cuuint64_t)cols / tc::kTileK};
    const cuuint64_t strides[3] = {(cuuint64_t)cols * 2, (cuuint64_t)gap, (cuuint64_t)tc::kTileK * 2};
    const cuuint32_t box[4] = {(cuuint32_t)tc::kTileK, (cuuint32_t)box_rows, 2, (cuuint32_t)box_kb};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    const CUresult r = encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptr), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return nullptr;
    return &(halves_cache[key] = m);
  }
  bool rows_ready[4] = {};  // tc_rows_kernel's forms: shared memory limit raised

  // pair kernel: CTA pairs that run at a time (0: not available, -1: not asked yet), scratch and flags of cut tiles
  int wide_pairs = -1;
  bool wide_ready[4][2] = {};                   // forms by K blocks of a stage: shared memory limit raised
  float* wide_scratch = nullptr;
  size_t wide_scratch_floats = 0;
  int* wide_flags = nullptr;
  int resid_clusters[5] = {0, 0, 0, 0, 0};     // clusters of that many pairs that run at a time (residual form); [0]: asked

  const CUtensorMap* get(const void* ptr, int rows, int cols, int box_rows, int box_kb = tc::kStageKb) {
    auto key = std::make_tuple(ptr, rows, cols, box_rows, box_kb);
    auto it = cache.find(key);
    if (it != cache.end()) return &it->second;
    CUtensorMap m;
    // (column within a K block, row, K block): stride of a row = its pitch, of a K block = 128 bytes
    const cuuint64_t dims[3] = {(cuuint64_t)tc::kTileK, (cuuint64_t)rows, (cuuint64_t)cols / tc::kTileK};
    const cuuint64_t strides[2] = {(cuuint64_t)cols * 2, (cuuint64_t)tc::kTileK * 2};
    const cuuint32_t box[3] = {(cuuint32_t)tc::kTileK, (cuuint32_t)box_rows, (cuuint32_t)box_kb};
    const cuuint32_t estr[3] = {1, 1, 1};
    const CUresult r = encode(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
                              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return nullptr;
    return &(cache[key] = m);
  }
};

// K ranges of tc_gemm_kernel's plain form for up to 128 rows, scratch permitting: nearly two CTAs per SM (7/8 of the slots measured best:
// one split fewer costs no bandwidth and saves partial sums), at least four 64-wide K blocks per CTA.  With several row blocks of 128 a CTA
// needs most of an SM's shared and tensor memory: one CTA per SM.
inline int tc_gemm_splits(const TcGemm* g, int tiles, int kblocks, int rows) {
  int splits = ((rows <= 128 ? 2 : 1) * g->sm_count * 7 / 8) / tiles;
  if (splits > kblocks / 4) splits = kblocks / 4;
  const int ks = rows <= 64 ? tc::kStageKb : 1;
  if (splits > (kblocks + ks - 1) / ks) splits = (kblocks + ks - 1) / ks;
  if (splits > 16) splits = 16;
  return splits < 1 ? 1 : splits;
}

}  // namespace amph
