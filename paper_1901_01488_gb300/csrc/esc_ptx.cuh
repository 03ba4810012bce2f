// PTX and bounded-wait helpers the kernels share.
#pragma once
#include <cuda_runtime.h>

#include "esc_internal.h"

namespace esc {

constexpr uint64_t kWaitLimitNs = 2000000000ull;   // 2 s per bounded wait
constexpr uint32_t FULL = 0xffffffffu;

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(
                   smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(unsigned long long *p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

__device__ __forceinline__ void raise_status(ScratchHdr *hdr, unsigned status) {
  atomicCAS(&hdr->status, 0u, status);
  atomicExch(&hdr->abort, 1u);
}
__device__ __forceinline__ bool aborted(const ScratchHdr *hdr) {
  return *(volatile const unsigned *)&hdr->abort != 0u;
}

// Warp-collective bounded wait for the phase of parity `parity` of an
// mbarrier: every lane must observe the completion itself (so that every lane
// has acquire ordering), the warp leaves together, and the decision to give
// up is lane 0's, broadcast.  With `abortable` the wait also gives up as
// soon as the launch is aborting (used for every wait that does not guard an
// in-flight bulk copy, so that one timeout cannot cascade into more).
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, ScratchHdr *hdr,
                                          uint64_t limit_ns = kWaitLimitNs, bool abortable = false) {
  bool seen = mbar_try_wait(bar, parity);
  if (__all_sync(FULL, seen)) return true;
  const uint64_t t0 = globaltimer();
  for (uint32_t it = 1;; ++it) {
    if (!seen) seen = mbar_try_wait(bar, parity);
    if (__all_sync(FULL, seen)) return true;
    if ((it & 63u) == 0) {
      int give_up = 0;
      if ((threadIdx.x & 31) == 0) give_up = (abortable && aborted(hdr)) ? 1 : (globaltimer() - t0 > limit_ns) ? 2 : 0;
      give_up = __shfl_sync(FULL, give_up, 0);
      if (give_up) {
        if (give_up == 2 && (threadIdx.x & 31) == 0) raise_status(hdr, ESC_ETIMEOUT);
        return false;
      }
    }
  }
}

// Warp-collective non-blocking test: true only if every lane observed it.
__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return __all_sync(FULL, ok != 0);
}

}  // namespace esc
