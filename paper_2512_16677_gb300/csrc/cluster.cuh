// cluster.cuh -- thread-block clusters: size, rank, barrier and a load from
// another CTA's shared memory.
#pragma once

#include <cstdint>

namespace qk {

__device__ __forceinline__ unsigned cluster_ctas() {
  unsigned n;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n));
  return n;
}
__device__ __forceinline__ unsigned cluster_cta() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// The word at the address of `p` (shared memory) in CTA `rank` of the cluster.
__device__ __forceinline__ unsigned cluster_load(const unsigned* p, unsigned rank) {
  unsigned v;
  asm volatile(
      "{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %1, %2;\n\t"
      "ld.shared::cluster.u32 %0, [a];\n\t}"
      : "=r"(v)
      : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank)
      : "memory");
  return v;
}

}  // namespace qk
