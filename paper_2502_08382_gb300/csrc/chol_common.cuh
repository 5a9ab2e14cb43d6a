// Device functions shared by the Cholesky kernels and the forward solve.
#pragma once
#include <cstdint>

#include "common.cuh"

namespace feti {
namespace {

__device__ __forceinline__ int pop_item(int* queue) {
  __shared__ int item;
  __syncthreads();
  if (threadIdx.x == 0) item = atomicAdd(queue, 1);
  __syncthreads();
  return item;
}

// Update block of child gc: a small child's lives in the CTA's small region, a split root's (a child factored
// by another task) in its hand-over slot, others on the stack.
__device__ __forceinline__ const double* child_update(const DevPlan& P, int gc, const double* stack,
                                                      const double* smallreg, const double* hand) {
  if (hand && P.sn_hoff[gc] >= 0) return hand + P.sn_hoff[gc];
  return P.sn_small[gc] ? smallreg + P.usm_ofs[gc] : stack + P.upd_ofs[gc];
}

}  // namespace
}  // namespace feti
