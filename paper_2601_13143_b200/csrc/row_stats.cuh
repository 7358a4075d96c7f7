// Softmax statistics of few scored rows: what the kernel that makes them (score_rows.cu) and those that read them share.
#pragma once

#include "common.cuh"

namespace fastav {

constexpr int kRowTileTokens = 64;  // tokens per (max, sum 2^(z - max)) pair of a scored row and head

// Some lanes of a warp, LANES of them side by side: a row's pairs -> one (all of those lanes).  Lane l takes the tiles l, l + LANES, .., eight loads in flight.  The whole warp comes here, lanes without a row with tiles = 0.
constexpr int kMergeLanes = 16;
__device__ __forceinline__ float2 merge_row_stats(const float2* pairs, int tiles, int lane) {
  constexpr int kEach = 8;
  float top = -INFINITY, sum = 0.f;
#pragma unroll 1
  for (int t0 = lane; t0 < tiles; t0 += kEach * kMergeLanes) {
    float2 v[kEach];
#pragma unroll
    for (int u = 0; u < kEach; ++u) v[u] = t0 + kMergeLanes * u < tiles ? chain_load(pairs + t0 + kMergeLanes * u) : make_float2(-INFINITY, 0.f);
    float next = top;
#pragma unroll
    for (int u = 0; u < kEach; ++u) next = fmaxf(next, v[u].x);
    const float ref = next == -INFINITY ? 0.f : next;
    sum *= exp2f(top - ref);
#pragma unroll
    for (int u = 0; u < kEach; ++u) sum += v[u].y * exp2f(v[u].x - ref);
    top = next;
  }
  __syncwarp();
  float all = top;
#pragma unroll
  for (int d = kMergeLanes / 2; d; d >>= 1) all = fmaxf(all, __shfl_xor_sync(0xFFFFFFFFu, all, d));
  sum = top > -INFINITY ? sum * exp2f(top - all) : 0.f;
#pragma unroll
  for (int d = kMergeLanes / 2; d; d >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
  return make_float2(all, sum);
}

// What a term's weights are made with, 2^(z - x) y: from the merged pair, which a sum of exponentials and a logarithm in fp32 would
// only round (2-norm error of the scores against 64 bits, mean over eight shapes: 2.7e-7 -> 2.3e-7), or from a log-sum-exp.  A row that sees no key adds 0.
__device__ __forceinline__ float2 weight_from_pair(float2 pair) { return pair.y > 0.f ? make_float2(pair.x, 1.0f / pair.y) : make_float2(INFINITY, 0.f); }
__device__ __forceinline__ float2 weight_from_lse(float lse2) { return make_float2(lse2, 1.f); }

// The sum over the terms (head, scored row: term i of a sequence is row i of its logits) of the weights, in that order, of TOKENS tokens
// `step` apart of which `have` exist.  kUnroll terms are asked for at a time, 32 loads; one running sum per token: whoever adds
// them up gets the same bits.
template <int TOKENS>
struct Weights {
  static constexpr int kUnroll = 32 / TOKENS;
  float v[kUnroll][TOKENS];
  __device__ __forceinline__ void fetch(const float* col, int step, int have, int i0, int terms, int stride) {
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
#pragma unroll
      for (int t = 0; t < TOKENS; ++t) v[u][t] = i0 + u < terms && t < have ? chain_load(col + (long long)(i0 + u) * stride + t * step) : -INFINITY;
  }
  __device__ __forceinline__ void add(const float2* weight, int i0, int terms, float (&total)[TOKENS]) const {
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      if (i0 + u < terms) {
        const float2 w = weight[i0 + u];
#pragma unroll
        for (int t = 0; t < TOKENS; ++t) total[t] += exp2f(v[u][t] - w.x) * w.y;
      }
  }
};

}  // namespace fastav
