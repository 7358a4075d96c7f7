// Host-side rules that need neither CUDA nor a GPU (plain C++, tested by themselves).
#pragma once

#include <cstddef>
#include <cstdint>

namespace fastav {

// [at, at + bytes) lies inside the range of `size` bytes that starts at `start`.
inline bool inside_range(uintptr_t at, size_t bytes, uintptr_t start, size_t size) {
  return at >= start && bytes <= size && at - start <= size - bytes;
}

constexpr int kPortableCluster = 8;  // what every device of the architecture can place
constexpr int kMaxCluster = 16;      // beyond the portable 8: allowed per kernel, and only where the GPCs at hand have the SMs

// Clusters of each size that run at once with one block per SM (cudaOccupancyMaxActiveClusters on a B200): a cluster's
// blocks share a GPC, and the GPCs hold 16 to 20 SMs.  Sixteen clusters of eight take two rounds, 20 us instead of 10.
constexpr int kAtOnce[kMaxCluster + 1] = {0, 148, 74, 45, 33, 26, 22, 15, 15, 15, 11, 7, 7, 7, 7, 7, 7};

// Blocks per sequence, a power of two up to `limit`: as many as have at least `slice` tokens each and still run at once (sixteen
// clusters of eight take two rounds where sixteen of four take one).
inline int cluster_blocks(int batch, int max_seqlen, int slice, int limit) {
  int blocks = limit;
  while (blocks > 1 && (batch > kAtOnce[blocks] || max_seqlen <= blocks / 2 * slice)) blocks /= 2;
  return blocks;
}

}  // namespace fastav
