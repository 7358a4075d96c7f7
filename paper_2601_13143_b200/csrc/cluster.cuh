// What the cluster kernels share: distributed shared memory, block-wide sums, the last step of the selection.
#pragma once

#include "common.cuh"
#include "host_rules.h"
#include "select_keys.cuh"
#include "sm100_ptx.cuh"

namespace fastav {

// ---- distributed shared memory ---------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t remote(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(ptx::smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void remote_store(uint32_t a, unsigned v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void remote_store2(uint32_t a, unsigned x, unsigned y) {  // 8-byte aligned
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void remote_store4(uint32_t a, uint4 v) {  // 16-byte aligned
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();  // the aligned form needs whole warps
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}

// ---- sums over the block's threads, with one barrier inside (warp_a: one word per warp) ----------------
// The sum over the threads above this one.
template <int WARPS>
__device__ __forceinline__ unsigned sum_above(unsigned own, unsigned* warp_a, int lane, int warp) {
  unsigned incl = own;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned t = __shfl_down_sync(0xFFFFFFFFu, incl, d);
    if (lane + d < 32) incl += t;
  }
  if (lane == 0) warp_a[warp] = incl;
  __syncthreads();
  unsigned above = incl - own;
#pragma unroll
  for (int w = 1; w < WARPS; ++w)
    if (w > warp) above += warp_a[w];
  return above;
}

// The sum over the threads before this one.
template <int WARPS>
__device__ __forceinline__ unsigned sum_before(unsigned own, unsigned* warp_a, int lane, int warp) {
  unsigned incl = own;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
    if (lane >= d) incl += t;
  }
  if (lane == 31) warp_a[warp] = incl;
  __syncthreads();
  unsigned before = incl - own;
#pragma unroll
  for (int w = 0; w < WARPS - 1; ++w)
    if (w < warp) before += warp_a[w];
  return before;
}

// Rank of list[tid] among the `count` keys of `list` by counting; the one whose rank range covers `remaining` is the
// threshold (equal keys all write the same two values).
__device__ __forceinline__ void rank_finish(const unsigned* list, int count, int remaining, int tid, unsigned* threshold, int* need_eq) {
  if (tid < count) {
    const unsigned mine = list[tid];
    int above = 0, not_below = 0;
#pragma unroll 4
    for (int i = 0; i < count; ++i) {
      const unsigned other = list[i];
      above += other > mine;
      not_below += other >= mine;
    }
    if (above < remaining && remaining <= not_below) {
      *threshold = mine;
      *need_eq = remaining - above;
    }
  }
}

}  // namespace fastav
