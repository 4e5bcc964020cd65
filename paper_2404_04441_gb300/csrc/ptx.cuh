// Inline-PTX helpers for sm_103a: shared-memory mbarriers, TMA tile loads,
// and bounded waits.
#pragma once

#include <cuda.h>
#include <cstdint>

namespace gbw {

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(count)
               : "memory");
}

// Make barrier initialisation visible to the async (TMA) proxy.
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar,
                                                      uint32_t bytes) {
  asm volatile(
      "mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
          smem_addr(bar)),
      "r"(bytes)
      : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// As mbar_try_wait, with the barrier's shared-space address.
__device__ __forceinline__ bool mbar_try_wait_s(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Wait for the barrier phase with the given parity (the barrier by its
// shared-space address). Gives up after about limit_ns of wall time (or a
// fixed iteration cap) and returns false.
__device__ __forceinline__ bool mbar_wait_bounded_s(uint32_t bar, uint32_t parity,
                                                    uint64_t limit_ns) {
  if (mbar_try_wait_s(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t i = 1; i < (1u << 28); ++i) {
    if (mbar_try_wait_s(bar, parity)) return true;
    if ((i & 1023u) == 0 && global_timer_ns() - t0 > limit_ns) return false;
  }
  return false;
}

__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar,
                                                  uint32_t parity,
                                                  uint64_t limit_ns) {
  return mbar_wait_bounded_s(smem_addr(bar), parity, limit_ns);
}

// As mbar_wait_bounded_s, for waits that the threads of a CTA take one by one
// and agree on later: a thread that gives up sets *failed (shared memory), and
// threads that still poll give up as soon as they see it.
__device__ __forceinline__ void mbar_wait_or_flag(uint32_t bar, uint32_t parity,
                                                  uint64_t limit_ns, volatile int *failed) {
  if (__builtin_expect(mbar_try_wait_s(bar, parity), 1)) return;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t i = 1; i < (1u << 28); ++i) {
    if (mbar_try_wait_s(bar, parity)) return;
    if ((i & 1023u) == 0 && (*failed || global_timer_ns() - t0 > limit_ns)) break;
  }
  *failed = 1;
}

// The wait of a CTA's ring for its stage s: every thread waits by itself, then
// one plain barrier. A stage that did not land is looked for every kRingLook
// stages (a barrier that carries a verdict costs more than a plain one) and,
// since the last stages need not be looked at, once more after the loop
// (ring_failed): true if this or an earlier stage gave up. Until then a CTA
// computes from what its slots hold; what it stores is void with the error.
constexpr int kRingLook = 3;

__device__ __forceinline__ bool ring_failed(volatile int *failed) {
  return __builtin_expect(*failed, 0);
}

__device__ __forceinline__ bool ring_wait(uint32_t bar, uint32_t parity, uint64_t limit_ns,
                                          volatile int *failed, bool look) {
  mbar_wait_or_flag(bar, parity, limit_ns, failed);
  __syncthreads();
  return look && ring_failed(failed);
}

// Waits, each within limit_ns, for the stages [first, end) of a ring of NB
// barriers, so that no TMA write lands in shared memory after the CTA exits.
template <int NB>
__device__ __forceinline__ void ring_drain(uint64_t *bars, int first, int end,
                                           uint64_t limit_ns) {
  for (int t = first; t < end; ++t) mbar_wait_bounded(&bars[t % NB], (t / NB) & 1, limit_ns);
}

// 3D tiled TMA load of one box into shared memory; completion is signalled
// on the barrier as transaction bytes. Coordinates are element indices
// (x innermost) and may lie outside the tensor: those elements read as zero.
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map,
                                            uint64_t *bar, int x, int y,
                                            int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_"
      "tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_addr(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_addr(bar)), "r"(x),
      "r"(y), "r"(z)
      : "memory");
}

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap *map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map))
               : "memory");
}

__device__ __forceinline__ float4 lds4(const float *p) {
  return *reinterpret_cast<const float4 *>(p);
}

}  // namespace gbw
