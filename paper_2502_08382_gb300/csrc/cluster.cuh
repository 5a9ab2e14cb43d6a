// Thread-block clusters: rank and size, barriers, and stores into another CTA's shared memory.
#pragma once
#include <cstdint>

#include "common.cuh"

namespace feti {
namespace {

__device__ __forceinline__ uint32_t cl_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cl_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// barrier of all threads of the cluster; orders their accesses to global and (distributed) shared memory
__device__ __forceinline__ void cl_barrier() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// v to the variable at `p` of CTA `rank`'s shared memory
__device__ __forceinline__ uint32_t cl_map(const void* p, int rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void cl_store(int* p, int rank, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cl_map(p, rank)), "r"(v) : "memory");
}
__device__ __forceinline__ void cl_store(double* p, int rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cl_map(p, rank)), "d"(v) : "memory");
}

}  // namespace
}  // namespace feti
