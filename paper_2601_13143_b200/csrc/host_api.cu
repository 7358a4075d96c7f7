// Host-buffer entry point: the same prune step for callers whose tensors live in host memory (offloaded activations / KV
// cache), all enqueued on the caller's stream and staged through a device arena the caller provides.
//
// Bound by PCIe, about 55 GB/s each way.  Where every buffer is page-locked the GPU can reach them itself, and two things
// follow.  Only what the method needs crosses the bus: K and the small arrays once, then the SURVIVORS' hidden states and
// V rows (the others are never uploaded).  And the two directions run at the same time: one kernel reads survivors' rows
// from host memory and writes them to the host outputs, instead of uploads, kernels and downloads in a row; a handful of
// copies of a few bytes each (2-4 us apiece) become part of two kernels.  2,048 tokens, half of them kept: 323 us
// instead of 636.
// Pageable buffers take the asynchronous copies.
#include <cuda.h>

#include "common.cuh"
#include "gather.cuh"
#include "host_rules.h"

namespace fastav {
namespace {

struct Arena {
  size_t q, q_idx, cu_qlens, k, v, cu_seqlens, lse, keep_counts, protect, hidden, pos;
  size_t scores, keep_idx, cu_keep, hidden_out, pos_out, k_out, v_out, status, workspace, workspace_bytes, total;
};

bool packed(const fastav_params& p) {
  const int64_t d = p.head_dim;
  return p.q_stride_head == d && p.q_stride_tok == d * p.num_q_heads && p.k_stride_head == d &&
         p.k_stride_tok == d * p.num_kv_heads && p.v_stride_head == d && p.v_stride_tok == d * p.num_kv_heads &&
         p.ko_stride_head == d && p.ko_stride_tok == d * p.num_kv_heads && p.vo_stride_head == d &&
         p.vo_stride_tok == d * p.num_kv_heads;
}

Arena plan_arena(const fastav_params& p) {
  Arena a{};
  size_t off = 0;
  auto carve = [&](size_t bytes) { const size_t at = off; off = align_up(off + bytes, 256); return at; };
  const size_t N = p.total_tokens, K = p.total_keep, B = p.batch, R = p.total_q;
  const size_t kv_row = (size_t)p.num_kv_heads * p.head_dim * 2;
  a.q = carve(R * p.num_q_heads * p.head_dim * 2);
  a.q_idx = carve(R * 4);
  a.cu_qlens = carve((B + 1) * 4);
  a.k = carve(N * kv_row);
  a.v = carve(N * kv_row);
  a.cu_seqlens = carve((B + 1) * 4);
  a.lse = carve(R * p.num_q_heads * 4);
  a.keep_counts = carve(B * 4);
  a.protect = carve(N);
  a.hidden = carve(N * (size_t)p.hidden * 2);
  a.pos = carve(N * 4);
  a.scores = carve(N * 4);
  a.keep_idx = carve(K * 4);
  a.cu_keep = carve((B + 1) * 4);
  a.hidden_out = carve(K * (size_t)p.hidden * 2);
  a.pos_out = carve(K * 4);
  a.k_out = carve(K * kv_row);
  a.v_out = carve(K * kv_row);
  a.status = carve(4);
  a.workspace_bytes = plan_workspace(p).total;
  a.workspace = carve(a.workspace_bytes);
  a.total = off;
  return a;
}

// ---- the page-locked path ----------------------------------------------------------------------------
constexpr int kCopyThreads = 256;
// Blocks of the gather through PCIe: a quarter of the SMs keeps enough rows on the way; more only crowd the link.  18 / 37 / 74 /
// 148 blocks, us per call: 2,048 tokens of 9 KB (hidden 3,584), 30 % kept 268 / 229 / 240 / 238, half 348 / 318 / 328 / 340, 90 % 494 / 505 /
// 516 / 534, 1,200 tokens of 12 KB, 40 % 262 / 231 / 240 / 242, 500 tokens of 9 KB, half 103 / 105 / 105 / 106, 2,048 of 1.5 KB 81 / 81 /
// 82 / 86, 400 of 1.5 KB 47 / 43 / 43 / 44.
constexpr int kHostGatherBlocks = kNumSMs / 4;
constexpr int kCopyUnroll = 8;                                   // 16-byte loads in flight per thread
constexpr int kPieceBytes = kCopyThreads * kCopyUnroll * 16;     // what a block copies at a time: 32 KB
constexpr int kMaxSegments = 12;

struct CopyList {
  struct {
    const unsigned char* src;
    unsigned char* dst;
    unsigned long long bytes;
  } seg[kMaxSegments];
  int count = 0;
  long long pieces = 0;
  void add(void* dst, const void* src, size_t bytes) {
    if (!src || !dst || !bytes) return;
    seg[count++] = {static_cast<const unsigned char*>(src), static_cast<unsigned char*>(dst), (unsigned long long)bytes};
    pieces += (long long)((bytes + kPieceBytes - 1) / kPieceBytes);
  }
};

// Piece `piece` of the list by one block: 16 bytes at a time where both sides allow it, else single bytes (only the ends of
// an array, or a small array of odd alignment).
__device__ __forceinline__ void copy_piece(const CopyList& list, long long piece) {
  int i = 0;
  for (; i < list.count; ++i) {
    const long long here = (long long)((list.seg[i].bytes + kPieceBytes - 1) / kPieceBytes);
    if (piece < here) break;
    piece -= here;
  }
  if (i == list.count) return;
  const unsigned char* src = list.seg[i].src + piece * kPieceBytes;
  unsigned char* dst = list.seg[i].dst + piece * kPieceBytes;
  const unsigned long long left = list.seg[i].bytes - piece * kPieceBytes;
  const int bytes = left < (unsigned long long)kPieceBytes ? (int)left : kPieceBytes;
  int done = 0;
  if (((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0) {
    const int quads = bytes / 16;
    uint4 v[kCopyUnroll];
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
      const int q = u * kCopyThreads + threadIdx.x;
      if (q < quads) v[u] = load_stream(reinterpret_cast<const uint4*>(src) + q);
    }
#pragma unroll
    for (int u = 0; u < kCopyUnroll; ++u) {
      const int q = u * kCopyThreads + threadIdx.x;
      if (q < quads) store_row(reinterpret_cast<uint4*>(dst) + q, v[u]);
    }
    done = quads * 16;
  }
  for (int at = done + threadIdx.x; at < bytes; at += kCopyThreads) dst[at] = chain_load(src + at);
}

// Host arrays -> arena; the status word starts at zero.
__global__ void __launch_bounds__(kCopyThreads) host_upload_kernel(CopyList list, int32_t* device_status, ChainHead head) {
  chain_enter(head);
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) *device_status = 0;
  for (long long piece = blockIdx.x; piece < list.pieces; piece += gridDim.x) copy_piece(list, piece);
}

// The survivors' rows (hidden states and V straight from host memory, K from the arena) and the small results -> host memory.
__global__ void __launch_bounds__(kCopyThreads) host_gather_kernel(Shapes s, RowStreams t, CopyList list, const int32_t* __restrict__ keep_idx,
                                                                   const int32_t* __restrict__ cu_keep,
                                                                   const int32_t* __restrict__ cu_seqlens) {
  chain_enter(s);
  pdl_wait();
  pdl_acquire(keep_idx);
  pdl_acquire(cu_keep);
  pdl_acquire(cu_seqlens);
  for (long long piece = blockIdx.x; piece < list.pieces; piece += gridDim.x) copy_piece(list, piece);
  const RowShape shape(s, t);
  const bool global_idx = (s.flags & FASTAV_KEEP_IDX_GLOBAL) != 0;
  const int rows = min(chain_load_cached(cu_keep + s.batch), s.total_keep);
  const int lane = threadIdx.x & 31, step = gridDim.x * (kCopyThreads / 32);
  for (int row = blockIdx.x * (kCopyThreads / 32) + (threadIdx.x >> 5); row < rows; row += step) {  // a warp per row
    int lo = 0, hi = s.batch;  // largest b with cu_keep[b] <= row
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (chain_load_cached(cu_keep + mid) <= row) lo = mid; else hi = mid;
    }
    const long long src = (global_idx ? 0ll : (long long)chain_load_cached(cu_seqlens + lo)) + chain_load(keep_idx + row);
    if (src < 0 || src >= s.total_tokens) continue;  // (the selection's own indices: cannot happen)
    if (lane == 0 && t.pos_in) t.pos_out[row] = chain_load(t.pos_in + src);
    copy_row<32, kCopyUnroll>(s, t, shape, src, row, lane);
  }
}

struct Range {
  const void* at;
  size_t bytes;
  bool overlaps(const Range& o) const {
    const uintptr_t a = reinterpret_cast<uintptr_t>(at), b = reinterpret_cast<uintptr_t>(o.at);
    return at && o.at && a < b + o.bytes && b < a + bytes;
  }
};

// The address under which the GPU reaches a page-locked host array, or nullptr.  The whole array has to lie inside the one
// page-locked allocation or registration that its first byte belongs to: an array whose two ends are page-locked may
// still have a gap between them that the GPU must not touch.
using PointerAttributeFn = CUresult (*)(void*, CUpointer_attribute, CUdeviceptr);
PointerAttributeFn pointer_attribute_fn() {
  static void* entry = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult res;
    if (cudaGetDriverEntryPoint("cuPointerGetAttribute", &p, cudaEnableDefault, &res) != cudaSuccess || res != cudaDriverEntryPointSuccess) p = nullptr;
    return p;
  }();
  return reinterpret_cast<PointerAttributeFn>(entry);
}
void* mapped(const void* host, size_t bytes) {
  cudaPointerAttributes first{};
  if (cudaPointerGetAttributes(&first, host) != cudaSuccess || first.type != cudaMemoryTypeHost || !first.devicePointer) {
    (void)cudaGetLastError();
    return nullptr;
  }
  const PointerAttributeFn attribute = pointer_attribute_fn();
  const CUdeviceptr at = reinterpret_cast<CUdeviceptr>(first.devicePointer);
  CUdeviceptr start = 0;
  size_t size = 0;
  if (!attribute || attribute(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, at) != CUDA_SUCCESS ||
      attribute(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, at) != CUDA_SUCCESS || !inside_range(at, bytes, start, size))
    return nullptr;
  return first.devicePointer;
}

}  // namespace
}  // namespace fastav

using namespace fastav;

extern "C" {

int32_t fastav_host_arena_bytes(const fastav_params* params, size_t* out_bytes) {
  size_t ws = 0;
  const int32_t rc = fastav_workspace_bytes(params, &ws);  // validates the shapes
  if (rc != FASTAV_OK) return rc;
  if (!out_bytes) return FASTAV_ERR_INVALID_ARG;
  if (!packed(*params)) return FASTAV_ERR_UNSUPPORTED;
  *out_bytes = plan_arena(*params).total;
  return FASTAV_OK;
}

int32_t fastav_prune_host(const fastav_params* params, const void* q, const int32_t* q_idx, const int32_t* cu_qlens,
                          const void* k, const void* v, const int32_t* cu_seqlens, const float* lse_opt,
                          const int32_t* keep_counts, const uint8_t* protect_opt, const void* hidden_in, const int32_t* pos_in,
                          float* scores_out, int32_t* keep_idx_out, int32_t* cu_keep_out, void* hidden_out, int32_t* pos_out,
                          void* k_out, void* v_out, int32_t* status_out, void* device_arena, size_t arena_bytes, void* stream) {
  size_t need = 0;
  int32_t rc = fastav_host_arena_bytes(params, &need);
  if (rc != FASTAV_OK) return rc;
  if (!device_arena || (reinterpret_cast<uintptr_t>(device_arena) & 255u) || arena_bytes < need) return FASTAV_ERR_WORKSPACE;
  if (!q_idx || !cu_qlens || !cu_seqlens || !keep_counts || !scores_out || !keep_idx_out || !cu_keep_out || !k || !q)
    return FASTAV_ERR_INVALID_ARG;
  if ((v == nullptr) != (v_out == nullptr) || (hidden_in == nullptr) != (hidden_out == nullptr) ||
      (pos_in == nullptr) != (pos_out == nullptr) || !k_out)
    return FASTAV_ERR_INVALID_ARG;
  // The index arrays are uploaded by this very call, so its first kernel must not start before earlier work on
  // the stream has completed: the chaining flag is not forwarded.
  fastav_params p = *params;
  p.flags &= ~FASTAV_CHAIN_CALLS;
  const Arena a = plan_arena(p);
  unsigned char* base = static_cast<unsigned char*>(device_arena);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t N = p.total_tokens, K = p.total_keep, B = p.batch, R = p.total_q;
  const size_t kv_row = (size_t)p.num_kv_heads * p.head_dim * 2;
  auto dev = [&](size_t off, const void* host) -> void* { return host ? base + off : nullptr; };
  // Everything the fused call would refuse is refused here, before the first copy is enqueued.
  rc = validate_prune(&p, base + a.q, (const int32_t*)(base + a.q_idx), (const int32_t*)(base + a.cu_qlens), base + a.k, dev(a.v, v),
                      (const int32_t*)(base + a.cu_seqlens), (const int32_t*)(base + a.keep_counts), dev(a.hidden, hidden_in),
                      (const int32_t*)dev(a.pos, pos_in), (const float*)(base + a.scores), (const int32_t*)(base + a.keep_idx),
                      (const int32_t*)(base + a.cu_keep), dev(a.hidden_out, hidden_out), (const int32_t*)dev(a.pos_out, pos_out),
                      base + a.k_out, dev(a.v_out, v_out), base + a.workspace, a.workspace_bytes);
  if (rc != FASTAV_OK) return rc;
  {
    // Every array page-locked (the row arrays on 16-byte boundaries, the positions on 4-byte ones): the GPU fetches and delivers them itself.  With
    // inputs that are also outputs the order matters, which only the copies below keep.
    const size_t hidden_row = (size_t)p.hidden * 2, q_bytes = R * p.num_q_heads * p.head_dim * 2;
    const Range ins[] = {{q, q_bytes}, {q_idx, R * 4}, {cu_qlens, (B + 1) * 4}, {k, N * kv_row}, {v, N * kv_row}, {cu_seqlens, (B + 1) * 4},
                         {lse_opt, R * p.num_q_heads * 4}, {keep_counts, B * 4}, {protect_opt, N}, {hidden_in, N * hidden_row}, {pos_in, N * 4}};
    const Range outs[] = {{scores_out, N * 4}, {keep_idx_out, K * 4}, {cu_keep_out, (B + 1) * 4}, {hidden_out, K * hidden_row},
                          {pos_out, K * 4}, {k_out, K * kv_row}, {v_out, K * kv_row}, {status_out, 4}};
    bool ok = true;
    for (const Range& i : ins)
      for (const Range& o : outs) ok = ok && !i.overlaps(o);
    auto at = [&](const void* host, size_t bytes) -> void* {
      if (!host || !ok) return nullptr;
      void* p = mapped(host, bytes);
      ok = p != nullptr;
      return p;
    };
    auto aligned_at = [&](const void* host, size_t bytes, uintptr_t alignment) -> void* {
      void* p = at(host, bytes);
      ok = ok && (reinterpret_cast<uintptr_t>(p) & (alignment - 1)) == 0;
      return p;
    };
    auto at16 = [&](const void* host, size_t bytes) { return aligned_at(host, bytes, 16); };
    CopyList up, down;
    RowStreams rows{};
    up.add(base + a.k, at16(k, N * kv_row), N * kv_row);
    rows.hidden_in = static_cast<const uint16_t*>(at16(hidden_in, N * hidden_row));
    rows.v_in = static_cast<const uint16_t*>(at16(v, N * kv_row));
    rows.hidden_out = static_cast<uint16_t*>(at16(hidden_out, K * hidden_row));
    rows.k_out = static_cast<uint16_t*>(at16(k_out, K * kv_row));
    rows.v_out = static_cast<uint16_t*>(at16(v_out, K * kv_row));
    rows.pos_out = static_cast<int32_t*>(aligned_at(pos_out, K * 4, 4));
    up.add(base + a.q, at(q, q_bytes), q_bytes);
    up.add(base + a.q_idx, at(q_idx, R * 4), R * 4);
    up.add(base + a.cu_qlens, at(cu_qlens, (B + 1) * 4), (B + 1) * 4);
    up.add(base + a.cu_seqlens, at(cu_seqlens, (B + 1) * 4), (B + 1) * 4);
    up.add(base + a.lse, at(lse_opt, R * p.num_q_heads * 4), R * p.num_q_heads * 4);
    up.add(base + a.keep_counts, at(keep_counts, B * 4), B * 4);
    up.add(base + a.protect, at(protect_opt, N), N);
    up.add(base + a.pos, at(pos_in, N * 4), N * 4);
    down.add(at(scores_out, N * 4), base + a.scores, N * 4);
    down.add(at(keep_idx_out, K * 4), base + a.keep_idx, K * 4);
    down.add(at(cu_keep_out, (B + 1) * 4), base + a.cu_keep, (B + 1) * 4);
    down.add(at(status_out, 4), base + a.status, 4);
    if (ok && K > 0) {
      rows.k_in = reinterpret_cast<const uint16_t*>(base + a.k);
      rows.pos_in = pos_in ? reinterpret_cast<const int32_t*>(base + a.pos) : nullptr;
      int32_t* status = reinterpret_cast<int32_t*>(base + a.status);
      const int32_t *d_cu_seqlens = reinterpret_cast<const int32_t*>(base + a.cu_seqlens);
      int32_t *d_keep_idx = reinterpret_cast<int32_t*>(base + a.keep_idx), *d_cu_keep = reinterpret_cast<int32_t*>(base + a.cu_keep);
      chain_begin(p.flags);
      const int grid = (int)(up.pieces < 2 * kNumSMs ? (up.pieces > 0 ? up.pieces : 1) : 2 * kNumSMs);
      cudaError_t e = launch_chained(host_upload_kernel, dim3(grid), dim3(kCopyThreads), 0, st, up, status, ChainHead{});
      count_launches(1);
      // The kernels that follow read the arrays this one uploads before their own wait, so the next one waits first too.
      chain_begin(p.flags);
      bool gathered = false;
      if (e == cudaSuccess)
        e = enqueue_selection(p, base + a.q, (const int32_t*)(base + a.q_idx), (const int32_t*)(base + a.cu_qlens), base + a.k, d_cu_seqlens,
                              (const float*)dev(a.lse, lse_opt), (const int32_t*)(base + a.keep_counts),
                              (const uint8_t*)dev(a.protect, protect_opt), nullptr, (float*)(base + a.scores), d_keep_idx, d_cu_keep,
                              base + a.workspace, status, st, &gathered);
      if (e == cudaSuccess) {
        e = launch_chained(host_gather_kernel, dim3(kHostGatherBlocks), dim3(kCopyThreads), 0, st, make_shapes(p), rows, down, (const int32_t*)d_keep_idx,
                           (const int32_t*)d_cu_keep, d_cu_seqlens);
        count_launches(1);
      }
      return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? FASTAV_OK : FASTAV_ERR_CUDA;
    }
  }
  cudaError_t e = cudaSuccess;
  auto h2d = [&](size_t off, const void* src, size_t bytes) {
    if (e == cudaSuccess && src && bytes) e = cudaMemcpyAsync(base + off, src, bytes, cudaMemcpyHostToDevice, st);
  };
  auto d2h = [&](void* dst, size_t off, size_t bytes) {
    if (e == cudaSuccess && dst && bytes) e = cudaMemcpyAsync(dst, base + off, bytes, cudaMemcpyDeviceToHost, st);
  };
  h2d(a.q, q, R * p.num_q_heads * p.head_dim * 2);
  h2d(a.q_idx, q_idx, R * 4);
  h2d(a.cu_qlens, cu_qlens, (B + 1) * 4);
  h2d(a.k, k, N * kv_row);
  h2d(a.v, v, N * kv_row);
  h2d(a.cu_seqlens, cu_seqlens, (B + 1) * 4);
  h2d(a.lse, lse_opt, R * p.num_q_heads * 4);
  h2d(a.keep_counts, keep_counts, B * 4);
  h2d(a.protect, protect_opt, N);
  h2d(a.hidden, hidden_in, N * (size_t)p.hidden * 2);
  h2d(a.pos, pos_in, N * 4);
  if (e == cudaSuccess) e = cudaMemsetAsync(base + a.status, 0, 4, st);
  if (e != cudaSuccess) return FASTAV_ERR_CUDA;
  rc = fastav_prune(&p, base + a.q, (const int32_t*)(base + a.q_idx), (const int32_t*)(base + a.cu_qlens), base + a.k,
                    dev(a.v, v), (const int32_t*)(base + a.cu_seqlens), (const float*)dev(a.lse, lse_opt),
                    (const int32_t*)(base + a.keep_counts),
                    (const uint8_t*)dev(a.protect, protect_opt), dev(a.hidden, hidden_in), (const int32_t*)dev(a.pos, pos_in),
                    (float*)(base + a.scores), (int32_t*)(base + a.keep_idx), (int32_t*)(base + a.cu_keep),
                    dev(a.hidden_out, hidden_out), (int32_t*)dev(a.pos_out, pos_out), base + a.k_out, dev(a.v_out, v_out),
                    base + a.workspace, a.workspace_bytes, (int32_t*)(base + a.status), stream);
  if (rc != FASTAV_OK) return rc;
  d2h(scores_out, a.scores, N * 4);
  d2h(keep_idx_out, a.keep_idx, K * 4);
  d2h(cu_keep_out, a.cu_keep, (B + 1) * 4);
  d2h(hidden_out, a.hidden_out, K * (size_t)p.hidden * 2);
  d2h(pos_out, a.pos_out, K * 4);
  d2h(k_out, a.k_out, K * kv_row);
  d2h(v_out, a.v_out, K * kv_row);
  d2h(status_out, a.status, 4);
  return e == cudaSuccess ? FASTAV_OK : FASTAV_ERR_CUDA;
}

}  // extern "C"
