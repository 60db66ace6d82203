// psl_async.cuh -- mbarriers, TMA bulk copies and the lookup helpers shared by the
// neighbourhood-score kernels (psl_hot.cu, psl_lin.cu).  GPU side only.
#pragma once
#include <cstdint>

#include "psl_device.cuh"
#include "psl_internal.h"

namespace psl {

// ---- TMA bulk copies and mbarriers (sm_90 and later) ----
__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(mbar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_inval(uint32_t mbar) {
  asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(bytes) : "memory");
}
// global -> shared bulk copy (16-byte aligned addresses, size a multiple of 16) signalling mbar
__device__ __forceinline__ void tma_load_1d(uint32_t dst, const void *src, uint32_t bytes, uint32_t mbar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(mbar)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred P1;\n mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n selp.b32 %0, 1, 0, P1;\n}"
      : "=r"(done)
      : "r"(mbar), "r"(parity)
      : "memory");
  return done != 0;
}
// bounded wait: false if the phase did not complete within the iteration limit
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t mbar, uint32_t parity, int limit = 1 << 20) {
  for (int it = 0; it < limit; it++)
    if (mbar_try_wait(mbar, parity)) return true;
  return false;
}

template <int OFF>
__device__ __forceinline__ float lds_at(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1+%2];" : "=f"(v) : "r"(addr), "n"(OFF));
  return v;
}
__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(mbar) : "memory");
}

// 5-bit field Q of w, times 4 (a byte offset in bits 2..6)
template <int Q>
__device__ __forceinline__ uint32_t field4(uint32_t w) {
  if constexpr (Q == 0)
    return (w << 2) & 0x7Cu;
  else
    return (w >> (5 * Q - 2)) & 0x7Cu;
}

__device__ __forceinline__ void flush2(float &hi, float &lo, float &a0, float &a1) {
  float blk = a0 + a1;
  a0 = a1 = 0.f;
  flush_block(hi, lo, blk);
}

// number of super-blocks sb >= 0 of a tile starting at kt0 with kt0 + 30 sb + off <= bound
__device__ __forceinline__ int sb_count(int bound, int kt0, int off, int nsb) {
  const int d = bound - kt0 - off;
  return d < 0 ? 0 : min(nsb, d / kSbK + 1);
}

}  // namespace psl
