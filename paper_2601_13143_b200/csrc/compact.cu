// Survivor gather: out[i] = in[source(i)] for hidden states, K, V and position ids.
//
// The step Section 2.2 ("Fine pruning") implies when it shrinks the token set layer after layer: the following
// layers only ever see the survivors, so their rows are packed into a dense layout.  It moves
// about 85-90 % of all bytes of a prune call and is bound by HBM bandwidth: each row (7-8 KB of
// hidden state, 1-2 KB each of K and V) is read once and written once with 16-byte accesses, the
// whole thread block walking one row so that every warp instruction covers 512 contiguous bytes.
//
// Main path: bulk asynchronous copies.  A row is a handful of contiguous segments (the hidden state,
// K and V of the token); each warp runs its own ring of row-sized shared-memory slots, one lane per
// segment issuing cp.async.bulk global -> shared (completion on an mbarrier) and then shared ->
// global, several rows in flight per warp and no register staging.  Rows whose segments are not
// 16-byte friendly, or too long for the ring, take the load/store kernel below.
#include <limits.h>

#include "common.cuh"
#include "gather.cuh"
#include "sm100_ptx.cuh"

namespace fastav {
namespace {

constexpr int kThreads = 256;
constexpr int kUnroll = 4;  // 16-byte loads in flight per thread

__global__ void __launch_bounds__(kThreads) compact_rows_kernel(Shapes s, RowStreams t, const int32_t* __restrict__ keep_idx,
                                                                const int32_t* __restrict__ cu_keep,
                                                                const int32_t* __restrict__ cu_seqlens,
                                                                int32_t* device_status) {
  chain_enter(s);
  pdl_wait();  // keep_idx and cu_keep are the previous kernel's output
  pdl_acquire(keep_idx);
  pdl_acquire(cu_keep);
  pdl_acquire(cu_seqlens);
  const RowShape shape(s, t);
  const bool global_idx = (s.flags & FASTAV_KEEP_IDX_GLOBAL) != 0;
  int rows = chain_load_cached(cu_keep + s.batch);
  if (rows > s.total_keep) rows = s.total_keep;  // never write past the caller's buffers

  for (int row = blockIdx.x; row < rows; row += gridDim.x) {
    int lo = 0, hi = s.batch;  // largest b with cu_keep[b] <= row
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (chain_load_cached(cu_keep + mid) <= row) lo = mid; else hi = mid;
    }
    const long long src = (global_idx ? 0ll : (long long)cu_seqlens[lo]) + chain_load(keep_idx + row);
    const long long dst = row;
    if (src < cu_seqlens[lo] || src >= cu_seqlens[lo + 1]) {  // an index outside its sequence: skip the row, report
      if (threadIdx.x == 0 && device_status) atomicOr(device_status, FASTAV_DEV_BAD_INDEX);
      continue;
    }
    if (threadIdx.x == 0 && t.pos_in) t.pos_out[dst] = t.pos_in[src];

    copy_row<kThreads, kUnroll>(s, t, shape, src, dst, threadIdx.x);
  }
}

// ---- bulk-copy path ---------------------------------------------------------------------------------
constexpr int kBulkStages = 4;          // row slots per warp
constexpr int kAhead = kBulkStages - 2; // rows loaded ahead of the one being stored
constexpr int kBulkMaxWarps = 8;
constexpr int kBulkSmemBudget = 200 * 1024;
// Shared memory that a block asks for at least: more than half of what an SM has, so that there is one block per SM and no block of the next
// call's first kernel comes to lie beside it.  That one's key loads want the L1 that is left where shared memory is split for it alone; beside
// blocks of 25 to 64 KB it started early on an SM split for those, or not, as it happened.  us with what the rows take / 64 KB /
// 116 KB: 8 x 120 rows of 6 KB, 70 % kept 22.6 / 18.5 / 18.3, 1 x 1,500 22.0 / 22.0 / 17.5, 16 x 120, half kept 24.6 / 20.8 / 19.7, 10 x 170 of 9 KB 18.0 /
// 16.3 / 15.6, 8 stages from 520 tokens of 12 KB 103.3 / 94.3 / 92.1.  (Of 400 shapes one lost: 12 x 90 rows of 12 KB, 30 % kept 16.1 / 16.1 / 16.8.)
// Short lists are gathered so soon that the next call's launch beside them is worth more: 5 stages from 2,000 tokens, rows of 1.5
// KB, 25 KB used 55.1 / 55.1 / 56.7.
constexpr size_t kBulkAlone = 116 * 1024;
size_t list_smem(size_t used) { return used > kBulkAlone ? used : used > 28 * 1024 ? kBulkAlone : 64 * 1024; }

__global__ void __launch_bounds__(kBulkMaxWarps * 32, 1)
compact_rows_bulk_kernel(Shapes s, RowStreams t, const int32_t* __restrict__ keep_idx, const int32_t* __restrict__ cu_keep,
                         const int32_t* __restrict__ cu_seqlens, int n_segments, int packed_k, int packed_v, int row_bytes, int slots,
                         int32_t* device_status) {
  extern __shared__ __align__(128) unsigned char bulk_smem[];
  __shared__ uint64_t full[kBulkMaxWarps][kBulkStages];
  chain_enter(s);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const uint32_t ring = ptx::smem_u32(bulk_smem) + (uint32_t)warp * slots * row_bytes;  // a warp with fewer rows than stages has that many slots
  Segment seg{};
  const bool active = lane < n_segments && make_segment(s, t, lane, packed_k != 0, packed_v != 0, seg);
  if (lane == 0) {
    for (int i = 0; i < kBulkStages; ++i) ptx::mbar_init(ptx::smem_u32(&full[warp][i]), n_segments);
    ptx::fence_barrier_init();
  }
  __syncwarp();
  const bool global_idx = (s.flags & FASTAV_KEEP_IDX_GLOBAL) != 0;
  pdl_wait();  // keep_idx and cu_keep are the previous kernel's output
  pdl_acquire(keep_idx);
  pdl_acquire(cu_keep);
  pdl_acquire(cu_seqlens);
  // Where this warp's rows come from.  The index words of its first rows are asked for all at once: the bounds of the sequences,
  // one per lane, and the tokens (one read for a row that does not exist is never used).  One after the other they were four trips to L2
  // ahead of the first copy, and more where the sequence of a row was searched for: a chain of 13 stages from 744 tokens 171 ->
  // 164 us, 1 x 2,048 tokens 24.2 -> 23.3, 32 ragged sequences of up to 8,192 tokens 314 -> 308.
  const int first = blockIdx.x * warps + warp, step = gridDim.x * warps;
  const bool by_lane = s.batch < 32;
  int keep_at = INT_MAX, seq_at = 0;  // by_lane: cu_keep and cu_seqlens of entry `lane`
  if (by_lane && lane <= s.batch) {
    keep_at = chain_load_cached(cu_keep + lane);
    seq_at = chain_load_cached(cu_seqlens + lane);
  }
  auto token_of = [&](int i) -> int {  // keep_idx of this warp's row i
    const long long row = first + (long long)i * step;
    return row < s.total_keep ? chain_load(keep_idx + row) : 0;
  };
  int token[kAhead];
#pragma unroll
  for (int i = 0; i < kAhead; ++i) token[i] = token_of(i);
  int rows = by_lane ? __shfl_sync(0xFFFFFFFFu, keep_at, s.batch) : chain_load_cached(cu_keep + s.batch);
  if (rows > s.total_keep) rows = s.total_keep;  // never write past the caller's buffers
  const int my_rows = first < rows ? (rows - first + step - 1) / step : 0;
  if (!by_lane || lane >= s.batch) keep_at = INT_MAX;

  // Source token of row i, whose entry of keep_idx is `idx`, or -1 for an index outside its sequence (row skipped, reported).
  auto source_of = [&](int i, int idx) -> long long {
    const int row = first + i * step;
    int from, end;  // of the row's sequence
    if (by_lane) {
      const int b = max(0, 31 - __clz(__ballot_sync(0xFFFFFFFFu, keep_at <= row)));  // the last one that starts at or before it
      from = __shfl_sync(0xFFFFFFFFu, seq_at, b);
      end = __shfl_sync(0xFFFFFFFFu, seq_at, b + 1);
    } else {
      int lo = 0, hi = s.batch;  // largest b with cu_keep[b] <= row
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (chain_load_cached(cu_keep + mid) <= row) lo = mid; else hi = mid;
      }
      from = chain_load_cached(cu_seqlens + lo);
      end = chain_load_cached(cu_seqlens + lo + 1);
    }
    const long long src = (global_idx ? 0ll : (long long)from) + idx;
    if (src < from || src >= end) {
      if (lane == 0 && device_status) atomicOr(device_status, FASTAV_DEV_BAD_INDEX);
      return -1;
    }
    return src;
  };
  // Issue the loads of row i into slot i % stages (all lanes call; one lane per segment copies).
  auto issue_load = [&](int i, long long src) {
    const uint32_t bar = ptx::smem_u32(&full[warp][i % kBulkStages]);
    if (!active) return;
    if (src < 0) {  // skipped row: the slot's barrier still completes its phase, so later rows keep their parity
      ptx::mbar_arrive(bar);
    } else {
      ptx::mbar_arrive_expect_tx(bar, seg.bytes);
      bulk_load(ring + (i % kBulkStages) * row_bytes + seg.slot_off, seg.in + src * seg.in_stride, seg.bytes, bar);
    }
  };

  int abort_flag = 0;
  unsigned loaded = 0;  // bit i % 32: row i has loads in flight or done (not skipped)
  // The first rows' positions, one per lane, are read beside the rows and written after the first of them: where a warp has a row
  // or two, each read and written in turn would add a trip to memory.
  long long first_src = -1;
#pragma unroll
  for (int i = 0; i < kAhead; ++i)
    if (i < my_rows) {
      const long long src = source_of(i, token[i]);
      issue_load(i, src);
      if (src >= 0) loaded |= 1u << i;
      if (lane == i) first_src = src;
    }
  const bool has_pos = t.pos_in && first_src >= 0;
  const int32_t first_pos = has_pos ? t.pos_in[first_src] : 0;
  for (int i = 0; i < my_rows; ++i) {
    // The slot of row i + kAhead last held row i - 2: its store must have finished reading shared memory.
    const int next = i + kAhead;
    if (next < my_rows) {
      bulk_wait_read<1>();
      // (the token is read here and not ahead: tokens of 32 rows at a time took the wait out and made the gathers of 4 x 6,554
      // tokens 109 -> 115 us, 32 sequences of up to 4,096 214 -> 222)
      const long long src = source_of(next, chain_load(keep_idx + first + (long long)next * step));
      issue_load(next, src);
      if (src >= 0) {
        loaded |= 1u << (next & 31);
        if (lane == 0 && t.pos_in) t.pos_out[first + (long long)next * step] = t.pos_in[src];
      } else {
        loaded &= ~(1u << (next & 31));
      }
    }
    if (loaded & (1u << (i & 31))) {
      const uint32_t bar = ptx::smem_u32(&full[warp][i % kBulkStages]);
      // One answer for the warp: source_of needs all lanes, and a bound shuffled from one that had left would be any number.
      if (!ptx::mbar_wait_warp(bar, (i / kBulkStages) & 1, &abort_flag)) {
        if (lane == 0 && device_status) atomicOr(device_status, FASTAV_DEV_WAIT_EXPIRED);
        int never = 0;  // the copies in flight write into this block's shared memory: they are waited for before it may exit
        for (int r = i; r <= min(next, my_rows - 1); ++r)
          if (loaded & (1u << (r & 31))) ptx::mbar_wait_bounded(ptx::smem_u32(&full[warp][r % kBulkStages]), (r / kBulkStages) & 1, &never);
        break;
      }
      if (active) bulk_store(seg.out + (long long)(first + i * step) * seg.out_stride, ring + (i % kBulkStages) * row_bytes + seg.slot_off, seg.bytes);
    }
    bulk_commit();  // one group per row, empty or not, so that the wait above always counts rows
    if (i == 0 && has_pos) t.pos_out[first + (long long)lane * step] = first_pos;
  }
  bulk_wait_all();  // the slots and the outputs are this kernel's until every store has landed
}

// ---- rows read ahead ----------------------------------------------------------------------------------
// Where shared memory holds all rows of a call, survivors or not, they need not wait for the selection: every warp reads some tokens' rows
// while the kernel before this one selects, and when that has ended asks for their places among the survivors and stores the rows that
// have one.  (That kernel lets this one start after its own wait: the rows are complete by then.)
// What it saves is a trip to memory for the list and one for the rows; what it costs is reading the dropped rows, beside a kernel that
// reads keys.  So it is taken where most rows stay (placed_compact_applies).
constexpr int kPlacedMaxSequences = 16;
static_assert(kPlacedMaxSequences <= 31, "bounds are kept one per lane");
constexpr int kPlacedLeastRow = 2048;  // bytes: shorter rows gain nothing (11 stages from 649 tokens, 1.5 KB: 104.6 -> 105.9 us)
__global__ void __launch_bounds__(kBulkMaxWarps * 32, 1)
compact_placed_kernel(Shapes s, RowStreams t, const int32_t* __restrict__ place, const int32_t* __restrict__ cu_seqlens, int n_segments, int packed_k, int packed_v,
                      int row_bytes, int slots, int32_t* device_status) {
  extern __shared__ __align__(128) unsigned char bulk_smem[];
  __shared__ uint64_t full[kBulkMaxWarps];
  chain_enter(s, cu_seqlens);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const uint32_t ring = ptx::smem_u32(bulk_smem) + (uint32_t)warp * slots * row_bytes, bar = ptx::smem_u32(&full[warp]);
  Segment seg{};
  const bool active = lane < n_segments && make_segment(s, t, lane, packed_k != 0, packed_v != 0, seg);
  if (lane == 0) {
    ptx::mbar_init(bar, 1);
    ptx::fence_barrier_init();
  }
  // Lane i has row i of the warp; it counts if it lies in a sequence as the selection sees it (a cut one's rest has no place).
  const int seq_at = lane <= s.batch ? chain_load(cu_seqlens + lane) : 0;
  const int row = blockIdx.x + gridDim.x * (warp + warps * lane);
  bool there = false;
  for (int b = 0; b < s.batch; ++b) {
    const Span seq = checked_words(__shfl_sync(0xFFFFFFFFu, seq_at, b), __shfl_sync(0xFFFFFFFFu, seq_at, b + 1), s.total_tokens, s.max_seqlen);
    there |= lane < slots && row >= seq.first && row < seq.first + seq.count;
  }
  const unsigned mine = __ballot_sync(0xFFFFFFFFu, there);
  if (lane == 0 && mine) ptx::mbar_arrive_expect_tx(bar, __popc(mine) * row_bytes);
  __syncwarp();
  for (unsigned left = mine; left; left &= left - 1) {
    const int i = __ffs(left) - 1;
    const long long src = __shfl_sync(0xFFFFFFFFu, row, i);
    if (active) bulk_load(ring + i * row_bytes + seg.slot_off, seg.in + src * seg.in_stride, seg.bytes, bar);
  }
  const int pos = there && t.pos_in ? chain_load(t.pos_in + row) : 0;
  pdl_wait();
  pdl_acquire(place);
  const int at = there ? chain_load(place + row) : -1;
  const unsigned kept = __ballot_sync(0xFFFFFFFFu, at >= 0 && at < s.total_keep);
  if (((kept >> lane) & 1u) && t.pos_in) t.pos_out[at] = pos;
  int abort_flag = 0;
  if (mine && !ptx::mbar_wait_warp(bar, 0, &abort_flag)) {
    if (lane == 0 && device_status) atomicOr(device_status, FASTAV_DEV_WAIT_EXPIRED);
    int never = 0;  // the copies in flight write into this block's shared memory: waited for once more
    ptx::mbar_wait_bounded(bar, 0, &never);
    return;
  }
  for (unsigned left = kept; left; left &= left - 1) {
    const int i = __ffs(left) - 1;
    const long long dst = __shfl_sync(0xFFFFFFFFu, at, i);
    if (active) bulk_store(seg.out + dst * seg.out_stride, ring + i * row_bytes + seg.slot_off, seg.bytes);
  }
  bulk_commit();
  bulk_wait_all();
}

struct PlacedPlan {
  int warps, slots;
  bool all_sms;
  long long bytes(int row_bytes) const { return (long long)warps * slots * row_bytes; }
  bool fits(int row_bytes) const { return slots <= 32 && bytes(row_bytes) <= kBulkSmemBudget; }
};
PlacedPlan placed_on(const Shapes& s, int row_bytes, int sms) {
  const int least = row_bytes > 2048 ? 16384 / row_bytes : 8;  // blocks of at least about 16 KB or 8 rows
  const int even = (s.total_tokens + sms - 1) / sms, per_block = even > least ? even : least;
  PlacedPlan p{};
  p.slots = (per_block + kBulkMaxWarps - 1) / kBulkMaxWarps;
  p.warps = p.slots > 0 ? (per_block + p.slots - 1) / p.slots : 0;
  return p;
}
// A block per SM, and none on the SMs that select if the others hold all rows: a block that has to wait for such an SM starts reading when the
// selection is over.  us on all SMs / on the others, 80 % kept: 1 x 1,700 rows of 12 KB 21.6 / 20.2, 2 x 800 18.2 / 17.7, 1 x 1,700 of 9 KB 17.3 /
// 16.2, 8 x 120 of 6 KB 19.4 / 18.7.  From three sequences on the others are fewer, and rings of more than 150 KB there the slower way (3 x 500 rows of
// 12 KB 16.7 / 17.2, 3 x 650 of 9 KB 15.5 / 16.1).
PlacedPlan placed_plan(const Shapes& s, int row_bytes) {
  const int others = kNumSMs - few_blocks(s);
  PlacedPlan p = placed_on(s, row_bytes, others > 0 ? others : 1);
  if (others >= kNumSMs / 2 && p.fits(row_bytes) && (s.batch <= 2 || p.bytes(row_bytes) <= kBulkSmemBudget * 3 / 4)) return p;
  p = placed_on(s, row_bytes, kNumSMs);
  p.all_sms = true;
  return p;
}

}  // namespace

cudaError_t launch_compact(const Shapes& s, const int32_t* keep_idx, const int32_t* cu_keep,
                           const int32_t* cu_seqlens, const void* hidden_in, void* hidden_out, const int32_t* pos_in,
                           int32_t* pos_out, const void* k_in, void* k_out, const void* v_in, void* v_out,
                           int32_t* device_status, cudaStream_t stream) {
  if (s.total_keep <= 0) return cudaSuccess;
  RowStreams t{static_cast<const uint16_t*>(hidden_in), static_cast<uint16_t*>(hidden_out),
               static_cast<const uint16_t*>(k_in),      static_cast<uint16_t*>(k_out),
               static_cast<const uint16_t*>(v_in),      static_cast<uint16_t*>(v_out),
               pos_in,                                  pos_out};
  const BulkPlan plan = bulk_plan(s, t);
  const int n_segments = plan.n_segments, row_bytes = plan.row_bytes;
  const int forced = (s.flags & FASTAV_COMPACT_PATH_MASK);
  if (forced != FASTAV_COMPACT_PATH_LOADSTORE && n_segments >= 1 && n_segments <= 32 && row_bytes > 0 &&
      kBulkStages * row_bytes <= kBulkSmemBudget) {
    int warps = kBulkSmemBudget / (kBulkStages * row_bytes);
    if (warps > kBulkMaxWarps) warps = kBulkMaxWarps;
    cudaError_t e =
        once_per_context([] { return cudaFuncSetAttribute(compact_rows_bulk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBulkSmemBudget); });
    if (e != cudaSuccess) return e;
    int blocks = (s.total_keep + warps - 1) / warps;
    if (blocks > kNumSMs) blocks = kNumSMs;
    // No deeper rings than a warp has rows.
    const int rows_per_warp = (s.total_keep + blocks * warps - 1) / (blocks * warps);
    const int slots = rows_per_warp < kBulkStages ? rows_per_warp : kBulkStages;
    const size_t smem = list_smem((size_t)warps * slots * row_bytes);
    e = launch_chained(compact_rows_bulk_kernel, dim3(blocks), dim3(warps * 32), smem, stream, s, t, keep_idx, cu_keep, cu_seqlens,
                       n_segments, (int)plan.packed_k, (int)plan.packed_v, row_bytes, slots, device_status);
    count_launches(1);
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  int blocks = kNumSMs * 8;
  if (blocks > s.total_keep) blocks = s.total_keep;
  const cudaError_t e = launch_chained(compact_rows_kernel, dim3(blocks), dim3(kThreads), 0, stream, s, t, keep_idx, cu_keep,
                                       cu_seqlens, device_status);
  count_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

// The share kept from which reading all rows pays, us by the list / ahead: 4 x 200 rows of 9 KB 30 % kept 11.7 / 12.1, half 12.5 / 12.1, 80 % 13.9 / 12.5; 1 x
// 1,000 half 13.9 / 12.9, 80 % 15.7 / 13.1; 8 x 120 half 14.8 / 14.7, 80 % 16.7 / 15.0.  One or two short sequences leave so much of the chip idle
// that it pays from the first survivor on (330 rows, 10 % kept 10.1 / 9.3), up to 6 MB of dropped rows (2,000 rows of 12 KB, 10 % kept,
// 22 MB: 17.3 / 21.0).  With more sequences the reads meet more of the selecting kernel's (8 x 230 rows of 12 KB, 30 % kept 15.5 / 18.1, 31 x 60, half
// 16.5 / 20.2), and where blocks have to wait for an SM at all, it is the slower way from five sequences on (10 x 170 rows of 9 KB, 80 % kept 15.6 / 18.3).
bool placed_compact_applies(const Shapes& s, const RowStreams& rows) {
  const BulkPlan plan = bulk_plan(s, rows);
  if ((s.flags & FASTAV_COMPACT_PATH_MASK) != 0 || s.batch > kPlacedMaxSequences || s.total_keep <= 0 || plan.row_bytes < kPlacedLeastRow || plan.n_segments > 32) return false;
  const PlacedPlan p = placed_plan(s, plan.row_bytes);
  if (!p.fits(plan.row_bytes)) return false;
  const long long kept = s.total_keep, all = s.total_tokens;
  if (p.all_sms && (s.batch > 4 || kept * 20 < all * 13)) return false;
  if (s.batch <= 2 && (all - kept) * plan.row_bytes <= 6ll << 20) return true;
  return s.batch <= 4 ? kept * 2 >= all : s.batch <= 8 ? kept * 5 >= all * 3 : kept * 4 >= all * 3;
}

cudaError_t launch_compact_placed(const Shapes& s, const RowStreams& rows, const int32_t* place, const int32_t* cu_seqlens, int32_t* device_status,
                                  cudaStream_t stream) {
  const BulkPlan plan = bulk_plan(s, rows);
  const PlacedPlan p = placed_plan(s, plan.row_bytes);
  cudaError_t e = once_per_context([] { return cudaFuncSetAttribute(compact_placed_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kBulkSmemBudget); });
  if (e != cudaSuccess) return e;
  const int per_block = p.warps * p.slots, blocks = (s.total_tokens + per_block - 1) / per_block;
  e = launch_chained(compact_placed_kernel, dim3(blocks), dim3(p.warps * 32), p.bytes(plan.row_bytes) > (long long)kBulkAlone ? (size_t)p.bytes(plan.row_bytes) : kBulkAlone, stream, s, rows, place, cu_seqlens,
                     plan.n_segments, (int)plan.packed_k, (int)plan.packed_v, plan.row_bytes, p.slots, device_status);
  count_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace fastav
