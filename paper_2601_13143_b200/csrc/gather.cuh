// One survivor's row: where its pieces lie, and its copy with 16-byte loads and stores.
#pragma once

#include "common.cuh"
#include "sm100_ptx.cuh"

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

struct BulkPlan {
  bool packed_k, packed_v;
  int n_segments, row_bytes;
};
// Every segment must be 16-byte friendly (it is: rows and strides are multiples of 8 elements), and there may be at most one per lane.
inline BulkPlan bulk_plan(const Shapes& s, const RowStreams& t) {
  BulkPlan p;
  p.packed_k = t.k_in && s.k_sh == s.dim && s.ko_sh == s.dim;
  p.packed_v = t.v_in && s.v_sh == s.dim && s.vo_sh == s.dim;
  p.n_segments = (t.hidden_in ? 1 : 0) + (t.k_in ? (p.packed_k ? 1 : s.hkv) : 0) + (t.v_in ? (p.packed_v ? 1 : s.hkv) : 0);
  p.row_bytes = row_bytes_of(s, t);
  return p;
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
// ---- rows by bulk asynchronous copies ----------------------------------------------------------------------
struct Segment {  // one contiguous piece of a row
  const unsigned char* in;
  unsigned char* out;
  long long in_stride, out_stride;  // bytes between consecutive tokens
  unsigned bytes, slot_off;         // size, offset inside the row slot
};

__device__ __forceinline__ void bulk_load(uint32_t dst_smem, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst_smem),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, uint32_t src_smem, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(reinterpret_cast<uint64_t>(dst)),
               "r"(src_smem), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Segment `idx` of a row: [hidden] [K: one piece if packed, else one per head] [V: likewise].
__device__ __forceinline__ bool make_segment(const Shapes& s, const RowStreams& t, int idx, bool packed_k, bool packed_v, Segment& seg) {
  unsigned off = 0;
  int at = 0;
  if (t.hidden_in) {
    if (idx == at) {
      seg = {reinterpret_cast<const unsigned char*>(t.hidden_in), reinterpret_cast<unsigned char*>(t.hidden_out),
             (long long)s.hidden * 2, (long long)s.hidden * 2, (unsigned)s.hidden * 2, off};
      return true;
    }
    ++at;
    off += s.hidden * 2;
  }
  if (t.k_in) {
    const int pieces = packed_k ? 1 : s.hkv;
    if (idx < at + pieces) {
      const int h = idx - at;
      seg = {reinterpret_cast<const unsigned char*>(t.k_in + (long long)h * s.k_sh), reinterpret_cast<unsigned char*>(t.k_out + (long long)h * s.ko_sh),
             s.k_st * 2, s.ko_st * 2, (unsigned)((packed_k ? s.hkv : 1) * s.dim * 2), off + (unsigned)h * s.dim * 2};
      return true;
    }
    at += pieces;
    off += s.hkv * s.dim * 2;
  }
  if (t.v_in) {
    const int pieces = packed_v ? 1 : s.hkv;
    if (idx < at + pieces) {
      const int h = idx - at;
      seg = {reinterpret_cast<const unsigned char*>(t.v_in + (long long)h * s.v_sh), reinterpret_cast<unsigned char*>(t.v_out + (long long)h * s.vo_sh),
             s.v_st * 2, s.vo_st * 2, (unsigned)((packed_v ? s.hkv : 1) * s.dim * 2), off + (unsigned)h * s.dim * 2};
      return true;
    }
  }
  return false;
}
#endif

}  // namespace fastav
