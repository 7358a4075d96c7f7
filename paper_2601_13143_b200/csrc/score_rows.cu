// Importance score, Eq. 4 (Section 2.2), for FEW scored rows on sequences that the few-rows kernel does not take (more than 2,048
// tokens): the paper's fine stage on what a long prompt's global stage left.  Q_last is one row per head, so Q K^T is a
// matrix-vector product and the step is bound by reading K once from HBM.
//
//   logits   : a persistent kernel; a unit is 64 tokens of one KV head.  One warp streams the units' keys with TMA through a ring of
//              128 KB, eight warps take a unit each and multiply it (mma.sync: up to eight query rows of the KV group per
//              instruction; the query rows come from L1).  Logits [Hq, R, N] (R: the sequence's own rows; base-2 units, -inf where the
//              causal mask hides the key) go to the workspace, and with them (max, sum 2^(z - max)) of every row over the unit's tokens.
//   the rest : log-sum-exp per row from those pairs, and per token the fixed-order sum over heads and rows -- by the kernel that
//              selects (select_long.cu), or by two small kernels where the scores alone are wanted or the terms are many.
//
// A prune call with one row on 4 x 6,554 tokens (Mistral-7B shapes, 70 % kept) takes 93.6 us instead of 109.4 with a tcgen05 kernel
// for the logits and one each for statistics, scores and selection (its logits 23.5 us, the keys' floor 8.3), 32 ragged sequences of
// 512 to 4,096 tokens 203 instead of 217.5.  Of the 12 us from the start to the last unit 1.9 are the sequences' bounds (cold), about
// 9 the keys.  Taken and put back: fragments straight from global memory, a block per tile (27 us: not enough bytes in flight);
// four warps (14 us: they are the bound); the first 8 or 16 units prefetched into L2 ahead of the bounds (97.5 -> 97.9, 98.6).
//
// The tiles of 64 tokens do not depend on the batch, and every key goes through the same arithmetic whatever its place in its
// tile: a sequence's scores depend on the sequence only, and equal keys get bit-equal scores.
#include <cuda.h>
#include <limits.h>

#include "common.cuh"
#include "key_fragment.cuh"
#include "row_stats.cuh"
#include "sm100_ptx.cuh"

namespace fastav {
namespace {

constexpr int kWarps = 8;                    // warps that multiply
constexpr int kThreads = 32 * (kWarps + 1);  // and one that streams the keys
constexpr int kSubBytes = kRowTileTokens * 128;  // 64 tokens of one 64-element column block
constexpr int kRingBytes = 128 * 1024;

template <int DIM>
struct RowsRing {
  static constexpr int kUnitBytes = DIM / 64 * kSubBytes, kStages = kRingBytes / kUnitBytes;
  // A stage has one warp that waits for it: a wait names a phase by its parity only, and a warp that came a round too early would take
  // the phase before for its own.
  static_assert(kStages % kWarps == 0);
};

// The batch's tiles of 64 tokens in one list.  Up to 32 sequences each lane of a warp knows one; beyond, shared memory has for every sequence its
// bounds and how many tiles come before it (of batches beyond kTable for every `step`-th), and a warp finds a tile's sequence in two looks of 32
// entries.  The list has to be exact, since every block takes an equal run of it: with every sequence given as many tiles as the longest one
// has, the real ones of 64 sequences, one of 20,000 tokens and 63 of 500, all fell to a few blocks (Mistral-7B shapes, one row: score call 49 us
// instead of 503, prune 205 instead of 656; 100 of 300 to 3,000 tokens 72 / 131 and 482 / 532).  Two kernels, since all of a large call's code comes
// from memory again: 4 x 6,554 tokens 93.6 us, with the table for every batch 95.6, with both in one kernel 95.0.
constexpr int kTable = 1024;
// Behind the ring, as large as the batch needs.
struct SharedList {
  int4* bounds;  // [entries] first token, tokens, first scored row, scored rows (step 1)
  int* ahead;    // entry e at e + e / 32: both looks are free of bank conflicts
  int* warp_sum;
};
__host__ __device__ inline int table_entries(int batch) {
  if (batch <= kTable) return batch;
  const int step = (batch + kTable - 1) / kTable;
  return (batch + step - 1) / step;
}
inline int table_bytes(int batch) { return table_entries(batch) * (int)(sizeof(int4) + sizeof(int)) + (table_entries(batch) / 32 + 1) * (int)sizeof(int); }

// A sequence without scored rows has none: nobody needs its keys (20 x 3,000 tokens, every second one without: 185 us instead of 196).
__device__ __forceinline__ int tiles_of(int tokens, int rows) { return rows > 0 ? (tokens + kRowTileTokens - 1) / kRowTileTokens : 0; }
__device__ __forceinline__ int sum_upto(int lane, int v) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xFFFFFFFFu, v, d);
    if (lane >= d) v += t;
  }
  return v;
}

// Up to 32 sequences: each lane knows one, and a vote of the warp finds a tile's.
struct LaneList {
  const Shapes& s;
  const SharedList sh;
  const int32_t *cu_seqlens, *cu_qlens;
  int lane;
  int4 mine{0, 0, 0, 0};  // this lane's sequence
  int upto = 0, total;    // tiles of the sequences up to and with it
  bool bad = false;
  int at = -1, first = 0, tok0 = 0, tokens = 0, row0 = 0, row_count = 0;
  __device__ LaneList(const Shapes& s_, const SharedList& sh_, const int32_t* cu_seqlens_, const int32_t* cu_qlens_, int lane_)
      : s(s_), sh(sh_), cu_seqlens(cu_seqlens_), cu_qlens(cu_qlens_), lane(lane_) {}
  // One warp per block asks for the bounds, the others read them from shared memory (all of them on a few lines of L2 cost a microsecond).
  __device__ void open(int warp) {
    if (warp == 0 && lane < s.batch) {
      const Span q = seq_span(s, cu_seqlens, lane), r = row_span(s, cu_qlens, lane);
      bad = q.bad || r.bad;
      sh.bounds[lane] = make_int4(q.first, q.count, r.first, r.count);
    }
    __syncthreads();
    if (lane < s.batch) mine = sh.bounds[lane];
    upto = sum_upto(lane, tiles_of(mine.y, mine.w));
    total = __shfl_sync(0xFFFFFFFFu, upto, 31);
  }
  __device__ void look_up(int t) {  // the whole warp; t < total
    if (t == at) return;
    at = t;
    const int b = __ffs(__ballot_sync(0xFFFFFFFFu, upto > t)) - 1, end = __shfl_sync(0xFFFFFFFFu, upto, b);
    tok0 = __shfl_sync(0xFFFFFFFFu, mine.x, b);
    tokens = __shfl_sync(0xFFFFFFFFu, mine.y, b);
    row0 = __shfl_sync(0xFFFFFFFFu, mine.z, b);
    row_count = __shfl_sync(0xFFFFFFFFu, mine.w, b);
    first = (t - (end - tiles_of(tokens, row_count))) * kRowTileTokens;
  }
};

// More.
struct TableList {
  const Shapes& s;
  const SharedList sh;
  const int32_t *cu_seqlens, *cu_qlens;
  int lane;
  int step, entries, total;
  bool bad = false;         // a sequence that this thread has seen was cut
  // of the tile looked up last, in all lanes
  int first = 0, tok0 = 0, tokens = 0, row0 = 0, row_count = 0;
  int begin = 0, end = 0;   // the tiles of its sequence
  __device__ TableList(const Shapes& s_, const SharedList& sh_, const int32_t* cu_seqlens_, const int32_t* cu_qlens_, int lane_)
      : s(s_), sh(sh_), cu_seqlens(cu_seqlens_), cu_qlens(cu_qlens_), lane(lane_) {}
  // All threads of the block.  Each bound is asked for by one thread of it (by all its warps: a microsecond on a few lines of L2).
  // (Loops kept as loops: of a large call every line of code comes from memory again.)
  __device__ void open(int warp) {
    step = s.batch <= kTable ? 1 : (s.batch + kTable - 1) / kTable;
    entries = table_entries(s.batch);
    const int each = (entries + kThreads - 1) / kThreads, e0 = min(entries, (int)threadIdx.x * each), e1 = min(entries, e0 + each);
    int sum = 0;
#pragma unroll 1
    for (int e = e0; e < e1; ++e) {
      sh.ahead[e + e / 32] = sum;
#pragma unroll 1
      for (int b = e * step; b < min(s.batch, (e + 1) * step); ++b) {
        const Span q = seq_span(s, cu_seqlens, b), r = row_span(s, cu_qlens, b);
        bad |= q.bad | r.bad;
        sum += tiles_of(q.count, r.count);
        sh.bounds[e] = make_int4(q.first, q.count, r.first, r.count);
      }
    }
    int before = sum_upto(lane, sum) - sum;
    if (lane == 31) sh.warp_sum[warp] = before + sum;
    if (entries > 32) {  // (else all of them are the first warp's)
      __syncthreads();
#pragma unroll 1
      for (int w = 0; w < warp; ++w) before += sh.warp_sum[w];
    }
#pragma unroll 1
    for (int e = e0; e < e1; ++e) sh.ahead[e + e / 32] += before;
    __syncthreads();
    total = 0;
#pragma unroll
    for (int w = 0; w <= kWarps; ++w) total += sh.warp_sum[w];
  }
  __device__ void look_up(int t) {  // the whole warp; t < total
    if (t < begin || t >= end) {    // another sequence: the last one that starts at or before it
      const unsigned coarse = __ballot_sync(0xFFFFFFFFu, lane * 32 < entries && sh.ahead[lane * 33] <= t);
      const int e0 = (31 - __clz(coarse)) * 32;
      const unsigned fine = __ballot_sync(0xFFFFFFFFu, e0 + lane < entries && sh.ahead[e0 + lane + e0 / 32] <= t);
      const int e = e0 + 31 - __clz(fine);
      begin = sh.ahead[e + e / 32];
      int4 v = sh.bounds[e];
      if (step > 1) v = among(e, t);
      tok0 = v.x;
      tokens = v.y;
      row0 = v.z;
      row_count = v.w;
      end = begin + tiles_of(tokens, row_count);
    }
    first = (t - begin) * kRowTileTokens;
  }
  // Beyond kTable sequences: tile t's among those of entry e, 32 of them at a time (after the kernel's wait).  Moves `begin` up to it.
  __device__ int4 among(int e, int t) {
    const int stop = min(s.batch, (e + 1) * step);
#pragma unroll 1
    for (int b0 = e * step; b0 < stop; b0 += 32) {
      const int b = b0 + lane;
      const Span q = b < stop ? seq_span<true>(s, cu_seqlens, b) : Span{0, 0, false}, r = b < stop ? row_span<true>(s, cu_qlens, b) : Span{0, 0, false};
      const int own = tiles_of(q.count, r.count), with = begin + sum_upto(lane, own);
      const unsigned behind = __ballot_sync(0xFFFFFFFFu, with > t);
      if (behind) {
        const int from = __ffs(behind) - 1;
        begin = __shfl_sync(0xFFFFFFFFu, with - own, from);
        return make_int4(__shfl_sync(0xFFFFFFFFu, q.first, from), __shfl_sync(0xFFFFFFFFu, q.count, from), __shfl_sync(0xFFFFFFFFu, r.first, from),
                         __shfl_sync(0xFFFFFFFFu, r.count, from));
      }
      begin = __shfl_sync(0xFFFFFFFFu, with, 31);
    }
    return make_int4(0, 0, 0, 0);
  }
};

template <int DIM, typename List>
__global__ void __launch_bounds__(kThreads, 1)
score_rows_kernel(const __grid_constant__ CUtensorMap k_map, Shapes s, const uint16_t* __restrict__ q, const int32_t* __restrict__ q_idx,
                  const int32_t* __restrict__ cu_qlens, const int32_t* __restrict__ cu_seqlens, float* __restrict__ logits,
                  float2* __restrict__ stats, int rq, int stat_tiles, int32_t* device_status) {
  using Ring = RowsRing<DIM>;
  extern __shared__ unsigned char smem_raw[];
  __shared__ uint64_t full[Ring::kStages], empty[Ring::kStages];
  __shared__ int warp_sum[kWarps + 1], abort_flag;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t ring = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  if (threadIdx.x == 0) {
    for (int i = 0; i < Ring::kStages; ++i) {
      ptx::mbar_init(ptx::smem_u32(&full[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&empty[i]), 1);
    }
    abort_flag = 0;
    ptx::fence_barrier_init();
    ptx::prefetch_tensormap(&k_map);
  }
  chain_enter_late(s, cu_seqlens, cu_qlens, q_idx);
  int4* const table = reinterpret_cast<int4*>(smem_raw + (ring - ptx::smem_u32(smem_raw)) + kRingBytes);
  List list(s, SharedList{table, reinterpret_cast<int*>(table + table_entries(s.batch)), warp_sum}, cu_seqlens, cu_qlens, lane);
  list.open(warp);
  const int units = list.total * s.hkv, each = units / (int)gridDim.x, more = units - each * (int)gridDim.x;  // (the host sees to it that they fit)
  const int begin = each * (int)blockIdx.x + min((int)blockIdx.x, more), count = each + ((int)blockIdx.x < more ? 1 : 0);
  pdl_wait();  // q and k may be what earlier work wrote; the logits may still be read by it
  pdl_acquire(q);
  if (blockIdx.x == 0 && list.bad && device_status) atomicOr(device_status, FASTAV_DEV_SHAPE_MISMATCH);

  if (warp == kWarps) {
    int it = 0;
    bool ok = true;
    for (; it < count; ++it) {
      const int stage = it % Ring::kStages;
      const int u = begin + it, t = u / s.hkv;
      list.look_up(t);
      ok = ptx::mbar_wait_warp(ptx::smem_u32(&empty[stage]), ((it / Ring::kStages) & 1) ^ 1u, &abort_flag);
      if (!ok) break;
      if (lane == 0) {
        const uint32_t bar = ptx::smem_u32(&full[stage]);
        ptx::mbar_arrive_expect_tx(bar, Ring::kUnitBytes);
#pragma unroll
        for (int sub = 0; sub < DIM / 64; ++sub)
          ptx::tma_load_3d(ring + stage * Ring::kUnitBytes + sub * kSubBytes, &k_map, sub * 64, u - t * s.hkv, list.tok0 + list.first, bar);
      }
      __syncwarp();
    }
    pdl_trigger();  // all loads have been issued
    if (!ok && lane == 0 && device_status) atomicOr(device_status, FASTAV_DEV_WAIT_EXPIRED);
    // The copies in flight write into this block's shared memory: they are waited for before it may exit, also where another warp gave up.
    int never = 0;
    for (int t = max(0, it - Ring::kStages); t < it; ++t)
      ptx::mbar_wait_bounded(ptx::smem_u32(&full[t % Ring::kStages]), (t / Ring::kStages) & 1, &never);
    return;
  }

  const int r8 = lane >> 2, t4 = lane & 3;  // of a fragment: token (and query row as an operand); pair of columns
  const bool causal = (s.flags & FASTAV_CAUSAL) != 0;
  for (int it = warp; it < count; it += kWarps) {
    const int stage = it % Ring::kStages;
    const int u = begin + it, t = u / s.hkv;
    const int head = u - t * s.hkv;
    list.look_up(t);
    const int m = min(list.tokens - list.first, kRowTileTokens), rows = min(list.row_count, rq), flat = rows * s.group;
    // Query row f of the KV group: scored row f / G, head f % G.  A lane's 16-byte pieces of a query row, and of a key: elements 64
    // sub + 16 t4 + 8 i (any order of the contraction will do as long as both operands have it; this one reads the
    // swizzled tile free of bank conflicts).
    uint4 qv[DIM / 32];
    auto fetch_q = [&](int f0) {
      const int f = f0 + r8, r = f / s.group;
      const uint4* const from = reinterpret_cast<const uint4*>(q + (long long)(list.row0 + r) * s.q_st + (long long)(head * s.group + f - r * s.group) * s.q_sh + t4 * 16);
#pragma unroll
      for (int i = 0; i < DIM / 32; ++i) qv[i] = f < flat ? chain_load_cached(from + i / 2 * 8 + i % 2) : make_uint4(0, 0, 0, 0);
    };
    fetch_q(0);
    int lim[2], out_row[2];
    auto columns = [&](int f0) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int f = f0 + t4 * 2 + e, r = f / s.group;
        out_row[e] = (head * s.group + f - r * s.group) * rows + r;
        lim[e] = f < flat ? min(m - 1, causal ? chain_load_cached(q_idx + list.row0 + r) - list.first : INT_MAX) : -1;
      }
    };
    columns(0);
    if (!ptx::mbar_wait_warp(ptx::smem_u32(&full[stage]), (it / Ring::kStages) & 1, &abort_flag)) {
      if (lane == 0 && device_status) atomicOr(device_status, FASTAV_DEV_WAIT_EXPIRED);
      return;
    }
    const uint32_t tile = ring + stage * Ring::kUnitBytes;
    for (int f0 = 0; f0 < flat; f0 += 8) {
      if (f0 > 0) {
        fetch_q(f0);
        columns(f0);
      }
      float acc[4][4];
#pragma unroll
      for (int frag = 0; frag < 4; ++frag) {
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[frag][c] = 0.f;
#pragma unroll
        for (int i = 0; i < DIM / 32; ++i) {
          const uint32_t at = tile + i / 2 * kSubBytes + (frag * 16 + r8) * 128 + (((2 * t4 + i % 2) ^ r8) << 4);
          const uint4 lo = ptx::ld_shared4(at), hi = ptx::ld_shared4(at + 8 * 128);
          mma_16x8x16(acc[frag], lo.x, hi.x, lo.y, hi.y, qv[i].x, qv[i].y);
          mma_16x8x16(acc[frag], lo.z, hi.z, lo.w, hi.w, qv[i].z, qv[i].w);
        }
      }
      if (f0 + 8 >= flat) ptx::mbar_arrive_warp(ptx::smem_u32(&empty[stage]), lane);  // the keys have been read
      float* const out = logits + list.tok0 + list.first + r8;
      float top[2] = {-INFINITY, -INFINITY}, sum[2] = {0.f, 0.f};
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float* const row = out + (long long)out_row[e] * s.total_tokens;
        const bool valid = f0 + t4 * 2 + e < flat;
#pragma unroll
        for (int c = 0; c < 8; ++c) {  // token 8 c + r8
          float& x = acc[c / 2][c % 2 * 2 + e];
          x = 8 * c + r8 <= lim[e] ? x * s.scale_log2 : -INFINITY;
          if (valid && 8 * c + r8 < m) row[8 * c] = x;
          top[e] = fmaxf(top[e], x);
        }
      }
#pragma unroll
      for (int d = 4; d < 32; d <<= 1) {
        top[0] = fmaxf(top[0], __shfl_xor_sync(0xFFFFFFFFu, top[0], d));
        top[1] = fmaxf(top[1], __shfl_xor_sync(0xFFFFFFFFu, top[1], d));
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float ref = top[e] == -INFINITY ? 0.f : top[e];
#pragma unroll
        for (int c = 0; c < 8; ++c) sum[e] += ptx::ex2_approx(acc[c / 2][c % 2 * 2 + e] - ref);
      }
#pragma unroll
      for (int d = 4; d < 32; d <<= 1) {
        sum[0] += __shfl_xor_sync(0xFFFFFFFFu, sum[0], d);
        sum[1] += __shfl_xor_sync(0xFFFFFFFFu, sum[1], d);
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int f = f0 + t4 * 2 + e, r = f / s.group;
        if (r8 == 0 && f < flat)
          stats[((long long)(list.row0 + r) * s.hq + head * s.group + f - r * s.group) * stat_tiles + list.first / kRowTileTokens] = make_float2(top[e], sum[e]);
      }
    }
  }
}

// Sixteen lanes per head, scored row and sequence: the tiles' pairs -> one, in the place of the first, and log2-sum-exp2 (+inf for a row that
// sees no key).
__global__ void __launch_bounds__(256) score_rows_lse_kernel(Shapes s, const int32_t* __restrict__ cu_qlens, const int32_t* __restrict__ cu_seqlens,
                                                             float2* __restrict__ stats, int rq, int stat_tiles, float* __restrict__ lse) {
  chain_enter(s);
  pdl_wait();
  pdl_acquire(stats);
  pdl_acquire(cu_qlens);
  pdl_acquire(cu_seqlens);
  const int i = blockIdx.x * (256 / kMergeLanes) + threadIdx.x / kMergeLanes, head = i / rq, r = i % rq, lane = threadIdx.x & (kMergeLanes - 1);
  const Span seq = seq_span<true>(s, cu_seqlens, blockIdx.y), qrows = row_span<true>(s, cu_qlens, blockIdx.y);
  const bool there = head < s.hq && r < qrows.count;
  const long long at = there ? (long long)(qrows.first + r) * s.hq + head : 0;
  const float2 v = merge_row_stats(stats + at * stat_tiles, there ? (seq.count + kRowTileTokens - 1) / kRowTileTokens : 0, lane);
  if (there && lane == 0) {
    stats[at * stat_tiles] = v;
    lse[at] = v.y > 0.f ? v.x + log2f(v.y) : INFINITY;
  }
}

// At least the batch's units; of larger batches at least what is listed of arrays whose sequences overlap, too.
long long most_units(const Shapes& s) {
  const long long tiles = s.batch > 32 ? (long long)((s.max_seqlen + kRowTileTokens - 1) / kRowTileTokens) * s.batch
                                       : (long long)s.total_tokens / kRowTileTokens + s.batch;
  return tiles * s.hkv;
}

template <int DIM, typename List>
cudaError_t run_with(const Shapes& s, const CUtensorMap& k_map, const uint16_t* q, const int32_t* q_idx, const int32_t* cu_qlens, const int32_t* cu_seqlens,
                float* logits, float2* stats, int stat_tiles, int32_t* device_status, cudaStream_t stream) {
  const int smem = kRingBytes + 1024 + table_bytes(s.batch);
  cudaError_t e = once_per_context([] {
    return cudaFuncSetAttribute(score_rows_kernel<DIM, List>, cudaFuncAttributeMaxDynamicSharedMemorySize, kRingBytes + 1024 + table_bytes(kTable));
  });
  if (e != cudaSuccess) return e;
  const long long units = most_units(s);
  count_launches(1);
  return launch_chained(score_rows_kernel<DIM, List>, dim3((unsigned)(units < kNumSMs ? units : kNumSMs)), dim3(kThreads), smem, stream, k_map, s, q, q_idx,
                        cu_qlens, cu_seqlens, logits, stats, s.max_qlen, stat_tiles, device_status);
}
template <int DIM, typename... Args>
cudaError_t run(const Shapes& s, Args... args) {
  return s.batch <= 32 ? run_with<DIM, LaneList>(s, args...) : run_with<DIM, TableList>(s, args...);
}

}  // namespace

cudaError_t launch_rows(const Shapes& s, const Workspace& w, const void* q, const int32_t* q_idx, const int32_t* cu_qlens, const void* k,
                        const int32_t* cu_seqlens, unsigned char* ws, int32_t* device_status, cudaStream_t stream, bool* used) {
  CUtensorMap k_map;
  *used = (s.flags & FASTAV_SCORE_PATH_MASK) == 0 && score_wide_applies(s) && s.max_qlen <= kNarrowMaxRows && s.max_qlen * s.group <= 128 && most_units(s) < INT_MAX &&
          encode_rows_map(k, s.dim, s.hkv, s.total_tokens, s.k_st, s.k_sh, 1, kRowTileTokens, &k_map);
  if (!*used) return cudaSuccess;
  const uint16_t* qq = static_cast<const uint16_t*>(q);
  float* logits = reinterpret_cast<float*>(ws + w.logits_off);
  float2* stats = reinterpret_cast<float2*>(ws + w.stats_off);
  return s.dim == 128 ? run<128>(s, k_map, qq, q_idx, cu_qlens, cu_seqlens, logits, stats, w.stat_tiles, device_status, stream)
                      : run<64>(s, k_map, qq, q_idx, cu_qlens, cu_seqlens, logits, stats, w.stat_tiles, device_status, stream);
}

cudaError_t launch_rows_lse(const Shapes& s, const Workspace& w, const int32_t* cu_qlens, const int32_t* cu_seqlens, unsigned char* ws,
                            cudaStream_t stream) {
  count_launches(1);
  return launch_chained(score_rows_lse_kernel, dim3((s.hq * s.max_qlen + 256 / kMergeLanes - 1) / (256 / kMergeLanes), s.batch), dim3(256), 0, stream, s, cu_qlens, cu_seqlens,
                        reinterpret_cast<float2*>(ws + w.stats_off), s.max_qlen, w.stat_tiles, reinterpret_cast<float*>(ws + w.lse_off));
}

}  // namespace fastav
