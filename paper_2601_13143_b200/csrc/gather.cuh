// One survivor's row: where its pieces lie, and its copy with 16-byte loads and stores.
#pragma once

#include "common.cuh"

namespace fastav {

struct RowStreams {
  const uint16_t* hidden_in;
  uint16_t* hidden_out;
  const uint16_t* k_in;
  uint16_t* k_out;
  const uint16_t* v_in;
  uint16_t* v_out;
  const int32_t* pos_in;
  int32_t* pos_out;
};

inline int row_bytes_of(const Shapes& s, const RowStreams& t) {
  return (t.hidden_in ? s.hidden * 2 : 0) + ((t.k_in ? 1 : 0) + (t.v_in ? 1 : 0)) * s.hkv * s.dim * 2;
}

#ifdef __CUDACC__
__device__ __forceinline__ uint4 load_stream(const uint4* p) {
  uint4 v;
  // a plain (coherent) load: under programmatic launch the rows may be what the previous kernel wrote
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

__device__ __forceinline__ void store_row(uint4* p, const uint4& v) {
  asm volatile("st.global.v4.u32 [%0], {%1,%2,%3,%4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// 16-byte chunks of a row: [hidden | K heads | V heads].
struct RowShape {
  int per_head, head_shift, n_hidden, n_k, n_chunks;
  __device__ __forceinline__ RowShape(const Shapes& s, const RowStreams& t) {
    per_head = s.dim >> 3;
    head_shift = s.dim == 128 ? 4 : 3;
    n_hidden = t.hidden_in ? s.hidden >> 3 : 0;
    n_k = t.k_in ? s.hkv * per_head : 0;
    n_chunks = n_hidden + n_k + (t.v_in ? s.hkv * per_head : 0);
  }
};

// Where chunk `c` of row `src` / `dst` lies.
__device__ __forceinline__ const uint4* chunk_in(const Shapes& s, const RowStreams& t, const RowShape& shape, long long src, int c) {
  if (c < shape.n_hidden) return reinterpret_cast<const uint4*>(t.hidden_in + src * s.hidden + (c << 3));
  c -= shape.n_hidden;
  const bool is_k = c < shape.n_k;
  if (!is_k) c -= shape.n_k;
  const int head = c >> shape.head_shift, off = (c & (shape.per_head - 1)) << 3;
  return reinterpret_cast<const uint4*>(is_k ? t.k_in + src * s.k_st + head * s.k_sh + off : t.v_in + src * s.v_st + head * s.v_sh + off);
}
__device__ __forceinline__ uint4* chunk_out(const Shapes& s, const RowStreams& t, const RowShape& shape, long long dst, int c) {
  if (c < shape.n_hidden) return reinterpret_cast<uint4*>(t.hidden_out + dst * s.hidden + (c << 3));
  c -= shape.n_hidden;
  const bool is_k = c < shape.n_k;
  if (!is_k) c -= shape.n_k;
  const int head = c >> shape.head_shift, off = (c & (shape.per_head - 1)) << 3;
  return reinterpret_cast<uint4*>(is_k ? t.k_out + dst * s.ko_st + head * s.ko_sh + off : t.v_out + dst * s.vo_st + head * s.vo_sh + off);
}

// Row `src` of the inputs -> row `dst` of the outputs by WIDTH threads, UNROLL 16-byte loads in flight each.
template <int WIDTH, int UNROLL>
__device__ __forceinline__ void copy_row(const Shapes& s, const RowStreams& t, const RowShape& shape, long long src, long long dst, int thread) {
  for (int base = thread; base < shape.n_chunks; base += WIDTH * UNROLL) {
    uint4 regs[UNROLL];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u)
      if (base + u * WIDTH < shape.n_chunks) regs[u] = load_stream(chunk_in(s, t, shape, src, base + u * WIDTH));
#pragma unroll
    for (int u = 0; u < UNROLL; ++u)
      if (base + u * WIDTH < shape.n_chunks) store_row(chunk_out(s, t, shape, dst, base + u * WIDTH), regs[u]);
  }
}
#endif

}  // namespace fastav
