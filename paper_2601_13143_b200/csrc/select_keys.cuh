// Order-preserving integer images of scores, shared by the selection kernels.
#pragma once

#include "common.cuh"

namespace fastav {

constexpr unsigned kProtectedKey = 0xFFFFFFFFu;
constexpr int kDirectMax = 256;  // a bucket of at most this many keys is finished by counting ranks, not by more passes

// fp32 -> uint32 with the same ordering as the float comparison (-0 and +0 compare equal).
__device__ __forceinline__ unsigned order_key(float x) {
  if (x == 0.0f) x = 0.0f;
  const unsigned u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

}  // namespace fastav
