// Keys as operands of mma.sync, straight from global memory: what the kernels for few scored rows share.
#pragma once

#include "common.cuh"

namespace fastav {

// One warp, 16 tokens of one KV head.  The contraction may run over head_dim in any order as long as both operands use
// the same one, so a lane's fragment registers of two k-steps are ONE 16-byte piece of a row (lane t of a quad: elements
// 32 i + 8 t ..): the loads are 64 contiguous bytes per row and instruction and nothing is staged or transposed.
template <int DIM>
struct KeyFragment {
  uint4 lo[DIM / 32], hi[DIM / 32];  // tokens lane / 4 and lane / 4 + 8
  __device__ __forceinline__ void load(const uint16_t* k, long long st, int tokens, int lane) {  // `tokens` exist from `k` on
    const int r = lane >> 2;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    const uint16_t* p = k + r * st + (lane & 3) * 8;
#pragma unroll
    for (int i = 0; i < DIM / 32; ++i) {
      lo[i] = r < tokens ? chain_load(reinterpret_cast<const uint4*>(p + i * 32)) : zero;
      hi[i] = r + 8 < tokens ? chain_load(reinterpret_cast<const uint4*>(p + 8 * st + i * 32)) : zero;
    }
  }
};

__device__ __forceinline__ void mma_16x8x16(float (&c)[4], unsigned a0, unsigned a1, unsigned a2, unsigned a3, unsigned b0, unsigned b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

}  // namespace fastav
