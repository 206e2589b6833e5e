// Asynchronous-copy building blocks shared by the kernels that stage
// operands through shared memory: mbarriers (bounded waits), L2 cache
// policies, bulk copies (cp.async.bulk) and tiled tensor copies
// (cp.async.bulk.tensor, TMA).
#pragma once

#include <cstdint>

#include <cuda.h>

#include "common.cuh"

namespace gbmg {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
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
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// bounded wait: false once one second has passed on the global timer (or
// after 2^24 polls, whichever comes first)
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  constexpr uint64_t kBudgetNs = 1000000000ull;
  const uint64_t t0 = global_ns();
  for (uint32_t it = 0; it < (1u << 24); ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255u) == 255u && global_ns() - t0 > kBudgetNs) return false;
  }
  return false;
}
// bounded wait of one role of a CTA: gives up when another role has set the
// CTA's abort flag, and sets the flag and the error word when its own second has
// passed, so that no role waits for one that has left
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity,
                                              volatile int* abort_flag, int* err) {
  constexpr uint64_t kBudgetNs = 1000000000ull;
  if (mbar_try_wait(bar, parity)) return true;  // the common case: no timer read
  const uint64_t t0 = global_ns();
  for (uint32_t it = 0;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if ((it & 255u) == 255u && global_ns() - t0 > kBudgetNs) {
      *abort_flag = 1;
      atomicOr(err, 1);
      return false;
    }
  }
}
// the same for a whole warp (all 32 lanes call it), with one answer for its
// lanes: each polls for itself, and a lane that gave up alone would leave the
// others waiting for it at the next warp-wide instruction
__device__ __forceinline__ bool wait_or_abort_warp(uint64_t* bar, uint32_t parity,
                                                   volatile int* abort_flag, int* err) {
  return __all_sync(0xffffffffu, wait_or_abort(bar, parity, abort_flag, err));
}
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
// L2 policy for data read exactly once (the link stream): evicted first, so
// the spinors that nine sites share stay resident
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
// L2 policy for data several CTAs read (a spinor serves nine sites)
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
// bulk copy global -> this CTA's shared memory, completing `bytes` of
// transaction on the mbarrier (16-byte aligned addresses, bytes % 16 == 0)
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint "
      "[%0], [%1], %2, [%3], %4;" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(pol)
      : "memory");
}

// the same copy with the default L2 policy
__device__ __forceinline__ void bulk_g2s_plain(void* dst, const void* src, uint32_t bytes,
                                               uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// tiled 5-D tensor copy global -> this CTA's shared memory (the box of
// `map` at coordinates c0..c4, innermost first), completing its bytes on
// the mbarrier; `map` lives in kernel-parameter space (__grid_constant__)
__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, int c0, int c1,
                                            int c2, int c3, int c4, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4),
      "r"(smem_u32(bar))
      : "memory");
}

// Host: a tiled 5-D FP32 tensor map over `base` (dims innermost first, the
// byte strides of dims 1..4, box extents), no interleave or swizzle.  The
// encoder comes from the driver through the runtime's entry-point query.
inline CUtensorMap make_map_5d(const void* base, const cuuint64_t dims[5],
                               const cuuint64_t strides[4], const cuuint32_t box[5]) {
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                              const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                              const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static Encode encode = [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    GB_CHECK(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000,
                                              cudaEnableDefault, &q));
    GB_REQUIRE(fn && q == cudaDriverEntryPointSuccess, MG_ERR_CUDA,
               "cuTensorMapEncodeTiled is not available");
    return reinterpret_cast<Encode>(fn);
  }();
  CUtensorMap m;
  const cuuint32_t unit[5] = {1, 1, 1, 1, 1};
  const CUresult r = encode(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, const_cast<void*>(base), dims,
                            strides, box, unit, CU_TENSOR_MAP_INTERLEAVE_NONE,
                            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  GB_REQUIRE(r == CUDA_SUCCESS, MG_ERR_ARG, "tensor map: cuTensorMapEncodeTiled rejected the layout");
  return m;
}

}  // namespace gbmg
