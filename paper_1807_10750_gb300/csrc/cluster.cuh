// Shared-memory addresses, cluster barriers and bounded mbarrier waits.
#pragma once

#include <cstdint>

#include "sweep.cuh"

namespace isingx {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// The address in block `rank` of the cluster that a has in this block.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}

// Every thread of every block of the cluster.
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

__device__ __forceinline__ bool map_try(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0u;
}

// The bounded wait for a phase of a local mbarrier whose first tries failed.
static __device__ __noinline__ bool map_wait(uint32_t bar, uint32_t parity, int* error, long long budget) {
  const long long t0 = global_ns();
  for (;;) {
    for (int it = 0; it < 16; ++it)
      if (map_try(bar, parity)) return true;
    if (ld_relaxed_s32(error) != 0) return false;
    if (global_ns() - t0 > budget) {
      atomicExch(error, 1);
      return false;
    }
  }
}

}  // namespace isingx
