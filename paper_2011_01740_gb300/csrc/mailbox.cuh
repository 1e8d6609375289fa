// mailbox.cuh -- messages between the warps of a team (rkck45_teams.cu, rkck45_relay.cu, df64.cu):
// a warp's lanes write to shared memory and one of them arrives on an mbarrier,
// whose phase the receiving warp awaits.  Waits are bounded.
#pragma once

#include "common.cuh"

namespace ens {

constexpr uint32_t kTeamWait = 1u << 24;  // polls of one wait

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// the warp's writes above are complete for whoever waits for this phase
__device__ __forceinline__ void post(unsigned long long* bar) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0)
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// wait for the next phase; `phase` is that barrier's phase count in this warp
__device__ __forceinline__ bool await(unsigned long long* bar, uint32_t& phase) {
  const uint32_t b = smem_addr(bar), parity = phase & 1u;
  ++phase;
  for (uint32_t k = 0; k < kTeamWait; ++k) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(b), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// a barrier whose phases end when `senders` warps have posted
__device__ __forceinline__ void init_bar(unsigned long long* bar, int senders) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(senders));
}
__device__ __forceinline__ void init_bars(unsigned long long* bar, int count) {
  for (int k = 0; k < count; ++k) init_bar(bar + k, 1);
}

}  // namespace ens
