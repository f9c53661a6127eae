// Device helpers of the thread-block-cluster kernels: ranks, cluster barrier, remote stores
// that complete the receiver's mbarrier, and the bounded wait for them (sm_103a).
#pragma once

#include "cluster_steps.cuh"
#include "tc_common.cuh"

namespace ddppo {

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// 16 bytes into another CTA's shared memory; they count towards its barrier's bytes
__device__ __forceinline__ void send16(uint32_t raddr, uint4 v, uint32_t rbar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
          raddr),
      "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(rbar)
      : "memory");
}
__device__ __forceinline__ void expect_bytes(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}
// bounded wait for the peers' bytes (acquire at cluster scope)
__device__ __forceinline__ bool wait_bytes(uint64_t* bar, uint32_t parity, int32_t* err) {
  for (uint32_t i = 0; i < TC_SPIN_LIMIT; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred P1;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 P1, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, P1;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    // a CTA elsewhere gave up: stop waiting for its bytes
    if ((i & 1023u) == 1023u && err && (*(volatile int32_t*)err & ERRF_TIMEOUT)) return false;
  }
  if (err) atomicOr(err, ERRF_TIMEOUT);
  return false;
}
__device__ __forceinline__ void send4(uint32_t raddr, float v, uint32_t rbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(raddr),
               "r"(__float_as_uint(v)), "r"(rbar)
               : "memory");
}

// After the last step. Every CTA tells the others the last step it sent and meets them: what
// is sent from here on is nothing. A CTA that gave up in step t may still be written to: its
// peers have sent step t, and those that had received all of it step t + 1. It waits (bounded)
// for these blocks before its shared memory goes away, counting the blocks that never come as
// delivered, so that the phase completes with the last one in flight.
constexpr int kClusterMax = 16;
__device__ __forceinline__ void cluster_end(uint64_t* full, int* sent, int ctas, int t, int T,
                                            uint32_t cta_bytes, bool failed) {
  __syncwarp();
  if ((int)threadIdx.x < ctas)
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(
                     map_rank(smem_addr(&sent[cluster_rank()]), threadIdx.x)),
                 "r"(min(t, T - 1))
                 : "memory");
  __syncwarp();
  cluster_sync();
  if (!failed || threadIdx.x != 0) return;
  for (int s = t; s <= t + 1; ++s) {
    const int missing = step_missing(sent, ctas, s, T);
    if (missing < 0) continue;
    uint64_t* bar = &full[step_bar(s)];
    if (missing)
      asm volatile("mbarrier.complete_tx.relaxed.cluster.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)),
                   "r"(missing * cta_bytes)
                   : "memory");
    mbar_drain_wait(bar, step_parity(s));
  }
}

}  // namespace ddppo
