// Importance score, Eq. 4 (Section 2.2), for MANY scored rows per sequence -- the tensor-core path.
//
// With R scored rows and G query heads per KV head, the logits of one KV head are a dense
// [R G, d] x [d, n] contraction: every K byte is reused by R G query rows, so it runs on the 5th-gen
// tensor cores (tcgen05.mma, operands in shared memory, fp32 accumulators in tensor memory) and is
// bound by the exponentials of the softmax, not by HBM.  The [R G, n] logits are never stored; two
// sweeps over K recompute them:
//
//   sweep 1 (S = Q K^T, TMEM lanes = query rows): each thread owns one row and keeps a running
//            (max, sum 2^(z - max)) over the key chunk of its block -> stats, merged into a
//            log2-sum-exp2 per (row, head);
//   sweep 2 (S^T = K Q^T, TMEM lanes = keys): each thread owns one key and adds 2^(z - lse) over 64 of
//            the block's query rows in a fixed column order; four such sums -> partial[KV head, row chunk][token];
//   finalize: scores = (sum of the partials in a fixed order) / (Hq R).
//
// One persistent block per SM works through its share of the units (sequence, KV head, chunk of up to 256
// query rows, chunk of key tiles); the share is computed on the device from cu_seqlens.  Warp 0 streams
// 128-key K tiles and the query tile with TMA (128-byte swizzle) through a 4-stage mbarrier ring, warp 1
// issues the MMAs into double-buffered accumulators, warps 2-17 (four warpgroups) read the accumulators
// back with tcgen05.ld and do the softmax arithmetic, part of the exponentials on the FMA pipe.
// The per-key arithmetic does not depend on the key's position, so equal keys get bit-equal scores; all
// sums have a fixed order, so runs are reproducible.  Every wait is bounded: a wait that expires makes the
// block give up, wait for its own copies, free its tensor memory and set FASTAV_DEV_WAIT_EXPIRED.
#include <cuda.h>

#include <limits.h>

#include "common.cuh"
#include "sm100_ptx.cuh"
#include "score_wide_math.cuh"

namespace fastav {
namespace {

constexpr int kTileKeys = 128;    // keys per K tile
constexpr int kRowsPerCta = 256;  // query rows (flat over scored row x head of the KV group) per block
constexpr int kStages = 4;        // K tiles in flight
constexpr int kGroups = 4;        // softmax warpgroups: four warps per scheduler hide each other's latencies
constexpr int kThreads = 64 + 128 * kGroups;  // warp 0: TMA, warp 1: MMA, warps 2-17: softmax
constexpr int kTmemCols = 512;
#ifndef FASTAV_UNITS_PER_BLOCK
#define FASTAV_UNITS_PER_BLOCK 7
#endif
constexpr int kUnitsPerBlock = FASTAV_UNITS_PER_BLOCK;  // aimed-at number of work units per block
constexpr int kMaxUnits = 48;       // work units one block may be given (the host sizes key chunks accordingly)
constexpr int kCtrlBytes = 18 * 1024;

template <int DIM>
struct Layout {
  static constexpr int kSubTiles = DIM / 64;                      // 128-byte-wide column blocks of a row
  static constexpr int kQSubBytes = kRowsPerCta * 128;            // one column block of the Q tile
  static constexpr int kKSubBytes = kTileKeys * 128;              // one column block of a K tile
  static constexpr int kQBytes = kSubTiles * kQSubBytes;
  static constexpr int kKTileBytes = kSubTiles * kKSubBytes;
  static constexpr int kQOff = 0;
  static constexpr int kKOff = kQOff + kQBytes;
  static constexpr int kCtrlOff = kKOff + kStages * kKTileBytes;  // barriers and small arrays
  static constexpr int kTotal = kCtrlOff + kCtrlBytes + 1024;     // + slack to align the base to 1024 bytes
};

using namespace widemath;
using ptx::tmem_ld_wait_for;

// What one block works on at a time: a run of K tiles of one (sequence, KV head, chunk of query rows).
struct Unit {
  int tok0, n;         // the sequence: first token in the packed batch, length
  int row0;            // first scored row of the sequence in q / q_idx
  int g, rc, kc;       // KV head, query-row chunk, key chunk
  int rows_here;       // query rows of the chunk that exist (a multiple of G)
  int new_q;           // the query tile differs from the previous unit's
};

constexpr int kKeptSpans = 64;
struct Control {
  uint64_t full_k[kStages], empty_k[kStages];
  uint64_t q_ready, q_free;
  uint64_t tmem_full[4], tmem_empty[4];
  uint64_t sums_ready[2];  // sweep 2: warpgroups 1-3 have published their partial sums of accumulator i
  uint32_t tmem_base;
  int abort;
  int n_units;
  int start_b, start_off;
  int warp_sums[kThreads / 32];
  int seq_first_unit[kThreads + 1];            // batch <= kThreads: first unit of every sequence, then the total
  alignas(16) float neg_lse[4 * kGroups][64];  // sweep 2, per softmax warp: -lse of its query-row columns (-inf: padding)
  alignas(16) int limit[4 * kGroups][64];      // sweep 2, per softmax warp: last key each column's row may see
  float sums[2][kGroups - 1][kTileKeys];       // sweep 2: per accumulator, the partial sums of warpgroups 1-3
  Span seqs[kKeptSpans], rows[kKeptSpans];     // of the first sequences: describing a unit needs them again
  Unit units[kMaxUnits];
};
static_assert(sizeof(Control) <= kCtrlBytes, "control block must fit its slot");

// Number of work units of sequence b: KV heads x query-row chunks x key chunks (0 for an empty sequence
// or one without scored rows).
__device__ __forceinline__ int units_of_spans(const Shapes& s, const Span& seq, const Span& rows, int rows_per_chunk, int chunk_keys) {
  const int n = seq.count, flat_rows = rows.count * s.group;
  if (n <= 0 || flat_rows <= 0) return 0;
  return s.hkv * ((flat_rows + rows_per_chunk - 1) / rows_per_chunk) * ((n + chunk_keys - 1) / chunk_keys);
}

// (through L1: for batches beyond the table, whose kernels wait first)
__device__ __forceinline__ int units_of_sequence(const Shapes& s, const int32_t* cu_seqlens, const int32_t* cu_qlens, int b,
                                                 int rows_per_chunk, int chunk_keys) {
  return units_of_spans(s, seq_span<true>(s, cu_seqlens, b), row_span<true>(s, cu_qlens, b), rows_per_chunk, chunk_keys);
}

// Block-wide sum of one int per thread (all threads get the result).
__device__ __forceinline__ int block_sum(int v, int* warp_sums) {
#pragma unroll
  for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, d);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = v;
  __syncthreads();
  int total = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) total += warp_sums[w];
  return total;
}

template <int DIM, int SWEEP>
__global__ void __launch_bounds__(kThreads, 1)
score_wide_kernel(const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap q_map, Shapes s,
                  const int32_t* __restrict__ q_idx, const int32_t* __restrict__ cu_qlens,
                  const int32_t* __restrict__ cu_seqlens, int chunk_tiles, int stat_chunks, int rc_max, int rows_per_chunk,
                  float2* __restrict__ stats, const float* __restrict__ lse, int lse_natural, float* __restrict__ partial,
                  int32_t* device_status) {
  using L = Layout<DIM>;
  extern __shared__ unsigned char smem_raw[];
  chain_enter_late(s, q_idx, cu_qlens, cu_seqlens);
  const uint32_t base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* base_ptr = smem_raw + (base - ptx::smem_u32(smem_raw));
  Control& ctl = *reinterpret_cast<Control*>(base_ptr + L::kCtrlOff);
  const uint32_t q_smem = base + L::kQOff, k_smem = base + L::kKOff;
  volatile int* abort = &ctl.abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk_keys = chunk_tiles * kTileKeys;
  const bool causal = (s.flags & FASTAV_CAUSAL) != 0;
  const int scored_per_chunk = rows_per_chunk / s.group;  // scored rows per query-row chunk (a multiple of 8)

  // ---- this block's share of the work: units [u0, u1) of the list ordered by (sequence, KV head,
  //      row chunk, key chunk), so that consecutive units mostly share their query tile -------------
  const bool table = s.batch <= kThreads;  // one sequence per thread: the unit table can be built in parallel
  int total_units = 0, my_units = 0, my_excl = 0;
  if (table) {
    const int b = threadIdx.x;
    if (b < s.batch) {
      const Span seq = seq_span(s, cu_seqlens, b), rows = row_span(s, cu_qlens, b);
      my_units = units_of_spans(s, seq, rows, rows_per_chunk, chunk_keys);
      if (b < kKeptSpans) {
        ctl.seqs[b] = seq;
        ctl.rows[b] = rows;
      }
    }
    int incl = my_units;  // inclusive scan inside the warp, then across warps through shared memory
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
      if (lane >= d) incl += t;
    }
    if (lane == 31) ctl.warp_sums[warp] = incl;
    __syncthreads();
    int warp_base = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
      if (w < warp) warp_base += ctl.warp_sums[w];
      total_units += ctl.warp_sums[w];
    }
    my_excl = warp_base + incl - my_units;
    ctl.seq_first_unit[b] = my_excl;  // first unit of sequence b in the global order
    if (b == 0) ctl.seq_first_unit[kThreads] = total_units;
  } else {
    pdl_wait();  // the bounds are read many times, one after the other below: after the wait, through L1
    pdl_acquire(cu_seqlens);
    pdl_acquire(cu_qlens);
    for (int b0 = 0; b0 < s.batch; b0 += kThreads) {
      const int b = b0 + threadIdx.x;
      total_units += block_sum(b < s.batch ? units_of_sequence(s, cu_seqlens, cu_qlens, b, rows_per_chunk, chunk_keys) : 0,
                               ctl.warp_sums);
    }
  }
  const int u0 = (int)((long long)total_units * blockIdx.x / gridDim.x);
  const int u1 = (int)((long long)total_units * (blockIdx.x + 1) / gridDim.x);
  if (u1 <= u0) {  // uniform: nothing for this block
    pdl_wait();
    return;
  }
  // The host sized the key chunks so that a block's share fits its table; a longer share means the device's
  // cu_seqlens describe more work than the host's total_tokens / batch did: the excess is left out and reported.
  const int n_mine = min(u1 - u0, kMaxUnits);
  if (threadIdx.x == 0 && u1 - u0 > kMaxUnits && device_status) atomicOr(device_status, FASTAV_DEV_SHAPE_MISMATCH);
  // Unit `target` of the global order -> what to work on.  `b` is its sequence, `off` its index inside it.
  auto describe = [&](int b, int off, Unit& un) {
    const bool kept = table && b < kKeptSpans;
    const Span seq = kept ? ctl.seqs[b] : table ? seq_span(s, cu_seqlens, b) : seq_span<true>(s, cu_seqlens, b);
    const Span rows = kept ? ctl.rows[b] : table ? row_span(s, cu_qlens, b) : row_span<true>(s, cu_qlens, b);
    if ((seq.bad || rows.bad) && device_status) atomicOr(device_status, FASTAV_DEV_SHAPE_MISMATCH);
    un.tok0 = seq.first;
    un.n = seq.count;
    un.row0 = rows.first;
    const int flat_rows = rows.count * s.group;
    const int row_chunks = (flat_rows + rows_per_chunk - 1) / rows_per_chunk;
    const int key_chunks = (un.n + chunk_keys - 1) / chunk_keys;
    const int grc = off / key_chunks;
    un.g = grc / row_chunks;
    un.rc = grc % row_chunks;
    un.kc = off % key_chunks;
    un.rows_here = min(rows_per_chunk, flat_rows - un.rc * rows_per_chunk);
    un.new_q = 1;
  };
  if (table) {
    __syncthreads();
    if (threadIdx.x < n_mine) {
      const int target = u0 + threadIdx.x;
      int lo = 0, hi = s.batch;  // smallest hi with first_unit[hi] > target; the sequence is hi - 1 (empty ones are skipped)
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        const int first_next = mid + 1 < s.batch ? ctl.seq_first_unit[mid + 1] : total_units;
        if (first_next > target) hi = mid; else lo = mid + 1;
      }
      Unit un;
      describe(lo, target - ctl.seq_first_unit[lo], un);
      ctl.units[threadIdx.x] = un;
    }
    __syncthreads();
    if (threadIdx.x > 0 && threadIdx.x < n_mine) {  // same sequence, KV head and row chunk as the unit before: same query tile
      const Unit &a = ctl.units[threadIdx.x - 1], &c = ctl.units[threadIdx.x];
      if (a.tok0 == c.tok0 && a.g == c.g && a.rc == c.rc) ctl.units[threadIdx.x].new_q = 0;
    }
  } else {
    int before = 0;  // units of the sequences before the current batch slice
    for (int b0 = 0; b0 < s.batch; b0 += kThreads) {
      const int b = b0 + threadIdx.x;
      const int mine = b < s.batch ? units_of_sequence(s, cu_seqlens, cu_qlens, b, rows_per_chunk, chunk_keys) : 0;
      int incl = mine;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int t = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += t;
      }
      __syncthreads();
      if (lane == 31) ctl.warp_sums[warp] = incl;
      __syncthreads();
      int warp_base = 0, slice_total = 0;
#pragma unroll
      for (int w = 0; w < kThreads / 32; ++w) {
        if (w < warp) warp_base += ctl.warp_sums[w];
        slice_total += ctl.warp_sums[w];
      }
      const int excl = before + warp_base + incl - mine;
      if (mine > 0 && excl <= u0 && u0 < excl + mine) {  // exactly one thread of one slice
        ctl.start_b = b;
        ctl.start_off = u0 - excl;
      }
      before += slice_total;
    }
    __syncthreads();
    if (threadIdx.x == 0) {  // very large batches: one thread walks this block's units
      int b = ctl.start_b, off = ctl.start_off;
      for (int i = 0; i < n_mine; ++i) {
        while (off >= units_of_sequence(s, cu_seqlens, cu_qlens, b, rows_per_chunk, chunk_keys)) {
          ++b;  // sequence exhausted (or empty): on to the next one
          off = 0;
        }
        Unit un;
        describe(b, off, un);
        if (i > 0 && ctl.units[i - 1].tok0 == un.tok0 && ctl.units[i - 1].g == un.g && ctl.units[i - 1].rc == un.rc) un.new_q = 0;
        ctl.units[i] = un;
        ++off;
      }
    }
  }
  if (threadIdx.x == 0) {
    const int count = n_mine;
    ctl.n_units = count;
    for (int i = 0; i < kStages; ++i) {
      ptx::mbar_init(ptx::smem_u32(&ctl.full_k[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl.empty_k[i]), 1);
    }
    ptx::mbar_init(ptx::smem_u32(&ctl.q_ready), 1);
    ptx::mbar_init(ptx::smem_u32(&ctl.q_free), 1);
    for (int i = 0; i < 4; ++i) {
      ptx::mbar_init(ptx::smem_u32(&ctl.tmem_full[i]), 1);
      // sweep 1: accumulator (e, i) is read by the two warpgroups of row tile e; sweep 2: accumulator i by all four
      ptx::mbar_init(ptx::smem_u32(&ctl.tmem_empty[i]), SWEEP == 1 ? 256 : 128 * kGroups);
    }
    for (int i = 0; i < 2; ++i) ptx::mbar_init(ptx::smem_u32(&ctl.sums_ready[i]), 128 * (kGroups - 1));
    ctl.abort = 0;
    ptx::fence_barrier_init();
    ptx::prefetch_tensormap(&k_map);
    ptx::prefetch_tensormap(&q_map);
  }
  // The query tile starts as zeros: rows no copy ever fills are then harmless operands.
  for (int i = threadIdx.x; i < L::kQBytes / 16; i += kThreads)
    asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(q_smem + i * 16), "r"(0) : "memory");
  ptx::fence_proxy_async_smem();  // ordered before the TMA writes that follow the barrier
  if (warp == 1) {
    ptx::tmem_alloc(ptx::smem_u32(&ctl.tmem_base), kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem = ctl.tmem_base;
  const int n_units = ctl.n_units;

  if (warp == 0) {
    // ---- TMA producer: one elected lane streams query tiles and K tiles ---------------------------
    if (lane == 0) {
      // q and k may be what the previous kernel in the stream wrote.  Sweep 2 may fetch them ahead of its wait: as a call's second
      // kernel, or as its first, which has waited already -- unless calls are chained (FASTAV_CHAIN_CALLS): then the previous
      // call's last kernel may still be running.
      if (SWEEP != 2 || (s.flags & FASTAV_CHAIN_CALLS)) pdl_wait();
      int tile_no = 0, q_gen = 0;  // K tiles / query tiles issued so far
      bool ok = true;
      for (int u = 0; u < n_units && ok; ++u) {
        const Unit un = ctl.units[u];
        if (un.new_q) {
          // The previous query tile must have been read by its last MMA before it is overwritten.
          if (q_gen > 0) ok = ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.q_free), (q_gen - 1) & 1, abort);
          if (!ok) break;
          // Boxes of 8 scored rows x G heads x 64 columns land as 8 G consecutive 128-byte rows, which is the
          // flat (scored row, head) order of the tile; 8 G rows are a whole number of 1024-byte swizzle groups.
          const int boxes = (un.rows_here / s.group + 7) / 8;
          const uint32_t box_bytes = 8u * s.group * 128u;
          const uint32_t bar = ptx::smem_u32(&ctl.q_ready);
          ptx::mbar_arrive_expect_tx(bar, boxes * box_bytes * L::kSubTiles);
          for (int sub = 0; sub < L::kSubTiles; ++sub)
            for (int i = 0; i < boxes; ++i)
              ptx::tma_load_3d(q_smem + sub * L::kQSubBytes + i * box_bytes, &q_map, sub * 64, un.g * s.group,
                               un.row0 + un.rc * scored_per_chunk + 8 * i, bar);
          ++q_gen;
        }
        const int key_begin = un.kc * chunk_keys;
        const int tiles = (min(un.n - key_begin, chunk_keys) + kTileKeys - 1) / kTileKeys;
        for (int t = 0; t < tiles; ++t, ++tile_no) {
          const int stage = tile_no % kStages;
          ok = ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.empty_k[stage]), ((tile_no / kStages) & 1) ^ 1u, abort);
          if (!ok) break;
          const uint32_t bar = ptx::smem_u32(&ctl.full_k[stage]);
          ptx::mbar_arrive_expect_tx(bar, L::kKTileBytes);
#pragma unroll
          for (int sub = 0; sub < L::kSubTiles; ++sub)
            ptx::tma_load_3d(k_smem + stage * L::kKTileBytes + sub * L::kKSubBytes, &k_map, sub * 64, un.g,
                             un.tok0 + key_begin + t * kTileKeys, bar);
        }
      }
      pdl_trigger();  // all loads have been issued
      if (*abort) {
        // Giving up: copies already issued still write into this block's shared memory, so wait (bounded
        // once more) for each of them before the block may exit.
        int never = 0;
        for (int t = max(0, tile_no - kStages); t < tile_no; ++t)
          ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.full_k[t % kStages]), (t / kStages) & 1, &never);
        if (q_gen > 0) ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.q_ready), (q_gen - 1) & 1, &never);
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer: one lane.  Issue by an elected lane of the whole warp is quicker, and so is one arrival per warp at the
    // accumulators' barriers, but these sweeps wait for their softmax warps, and both made them slower: 4 x 16,384 tokens, 128
    // rows, sweep 1 / 2: 86.3 / 80.0 us as it is, 87.0 / 80.9 with warp arrivals, 88.1 / 81.5 with elected issue, 90.0 / 82.0
    // with both.
    if (lane == 0) {
      int tile_no = 0, q_gen = 0;
      int uses0 = 0, uses1 = 0;  // sweep 1: how often the accumulators of 128-row tile e have been used
      bool ok = true;
      for (int u = 0; u < n_units && ok; ++u) {
        const Unit un = ctl.units[u];
        if (un.new_q) {
          ok = ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.q_ready), q_gen & 1, abort);
          if (!ok) break;
          ptx::tc_fence_after_sync();
          ++q_gen;
        }
        const int key_begin = un.kc * chunk_keys;
        const int tiles = (min(un.n - key_begin, chunk_keys) + kTileKeys - 1) / kTileKeys;
        const int mtiles = (un.rows_here + 127) / 128;     // sweep 1: 128-row MMA tiles in use
        const int n_cols = (un.rows_here + 31) / 32 * 32;  // sweep 2: MMA N (query rows as columns)
        for (int t = 0; t < tiles && ok; ++t, ++tile_no) {
          const int stage = tile_no % kStages;
          ok = ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.full_k[stage]), (tile_no / kStages) & 1, abort);
          if (!ok) break;
          const uint32_t k_tile = k_smem + stage * L::kKTileBytes;
          if constexpr (SWEEP == 1) {
            // S = Q K^T: A = 128 query rows, B = 128 keys; accumulator (e, i) at columns i*256 + e*128.
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              if (e >= mtiles || !ok) break;
              const int uses = e == 0 ? uses0 : uses1;
              const int i = uses & 1;
              ok = ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.tmem_empty[i * 2 + e]), ((uses >> 1) & 1) ^ 1u, abort);
              if (!ok) break;
              ptx::tc_fence_after_sync();
              ptx::umma_bf16_steps<DIM / 16, L::kQSubBytes, L::kKSubBytes, false>(tmem + i * 256 + e * 128, ptx::umma_desc_sw128(q_smem + e * 128 * 128, 0),
                                                                           ptx::umma_desc_sw128(k_tile, 0), ptx::umma_idesc_bf16(128, kTileKeys), false);
              ptx::umma_commit<false>(ptx::smem_u32(&ctl.tmem_full[i * 2 + e]));
              if (e == 0) ++uses0; else ++uses1;
            }
            if (!ok) break;
            ptx::umma_commit<false>(ptx::smem_u32(&ctl.empty_k[stage]));
          } else {
            // S^T = K Q^T: A = 128 keys, B = n_cols query rows; accumulator i at columns i*256.
            const int i = tile_no & 1;
            ok = ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.tmem_empty[i]), ((tile_no >> 1) & 1) ^ 1u, abort);
            if (!ok) break;
            ptx::tc_fence_after_sync();
            const uint32_t idesc = ptx::umma_idesc_bf16(kTileKeys, n_cols);
            ptx::umma_bf16_steps<DIM / 16, L::kKSubBytes, L::kQSubBytes, false>(tmem + i * 256, ptx::umma_desc_sw128(k_tile, 0), ptx::umma_desc_sw128(q_smem, 0),
                                                                         idesc, false);
            ptx::umma_commit<false>(ptx::smem_u32(&ctl.empty_k[stage]));
            ptx::umma_commit<false>(ptx::smem_u32(&ctl.tmem_full[i]));
          }
        }
        // Once the MMAs issued so far are done, the query tile may be replaced.
        if (ok && u + 1 < n_units && ctl.units[u + 1].new_q) ptx::umma_commit<false>(ptx::smem_u32(&ctl.q_free));
      }
    }
  } else {
    // ---- softmax warps: four warpgroups, so that every scheduler has four of them to pick from ---------
    const int wg = (warp - 2) >> 2;           // warpgroup 0..3
    const int quarter = warp & 3;             // the 32 TMEM lanes this warp may read
    const int my_lane = quarter * 32 + lane;  // row (sweep 1) or key (sweep 2) inside the tile
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
    pdl_wait();  // before the first read of lse (sweep 2) and the first write of stats / partial
    pdl_acquire(lse);
    pdl_acquire(q_idx);

    if constexpr (SWEEP == 1) {
      // Warpgroup (e, h) owns the rows of 128-row tile e and the keys [64 h, 64 h + 64) of every K tile:
      // thread <-> row, its running (max, sum) over that half of the keys -> one stats entry per half.
      const int e = wg & 1, h = wg >> 1;
      int uses = 0;
      bool ok = true;
      for (int u = 0; u < n_units && ok; ++u) {
        const Unit un = ctl.units[u];
        if (e * 128 >= un.rows_here) continue;  // this 128-row tile is not in use for the unit
        const int key_begin = un.kc * chunk_keys;
        const int tiles = (min(un.n - key_begin, chunk_keys) + kTileKeys - 1) / kTileKeys;
        const int f = un.rc * rows_per_chunk + e * 128 + my_lane;
        const bool row_valid = e * 128 + my_lane < un.rows_here;
        const int r = row_valid ? f / s.group : 0;
        const int last_visible = min(un.n - 1, (causal && row_valid) ? chain_load_cached(q_idx + un.row0 + r) : INT_MAX);
        float zmax = -INFINITY;
        float2 sum2 = make_float2(0.f, 0.f);
        for (int t = 0; t < tiles; ++t, ++uses) {
          const int i = uses & 1;
          ok = ptx::mbar_wait_warp(ptx::smem_u32(&ctl.tmem_full[i * 2 + e]), (uses >> 1) & 1, abort);
          if (!ok) break;
          ptx::tc_fence_after_sync();
          const int bound = last_visible - (key_begin + t * kTileKeys + h * 64);  // columns 0..bound of this half are visible
          const uint32_t taddr = lane_addr + i * 256 + e * 128 + h * 64;
          uint32_t va[32], vb[32];
          ptx::tmem_ld32(taddr, va);
          tmem_ld_wait_for(va);
          ptx::tmem_ld32(taddr + 32, vb);
          fold_row_piece_any(va, bound, s.scale_log2, zmax, sum2);
          tmem_ld_wait_for(vb);
          ptx::tc_fence_before_sync();
          ptx::mbar_arrive(ptx::smem_u32(&ctl.tmem_empty[i * 2 + e]));  // the accumulator may be overwritten
          fold_row_piece_any(vb, bound - 32, s.scale_log2, zmax, sum2);
        }
        if (ok && row_valid) {
          const long long rh = (long long)(un.row0 + r) * s.hq + un.g * s.group + f % s.group;
          stats[rh * stat_chunks + un.kc * 2 + h] = make_float2(zmax * s.scale_log2, sum2.x + sum2.y);
        }
      }
    } else {
      // Every K tile is shared by the four warpgroups: thread <-> key, warpgroup w sums the query-row columns
      // [64 w, 64 w + 64); warpgroups 1-3 publish their sums in shared memory and warpgroup 0 adds them in a
      // fixed order and writes the partial.  Each warp keeps its own copy of the per-column -lse and mask
      // limits (no block-level barrier between softmax warps).
      int tile_no = 0, min_limit = INT_MAX;
      bool ok = true;
      float* neg_lse = ctl.neg_lse[warp - 2];
      int* limit = ctl.limit[warp - 2];
      for (int u = 0; u < n_units && ok; ++u) {
        const Unit un = ctl.units[u];
        const int key_begin = un.kc * chunk_keys;
        const int tiles = (min(un.n - key_begin, chunk_keys) + kTileKeys - 1) / kTileKeys;
        const int my_cols = max(0, min(64, un.rows_here - wg * 64));  // columns of this warpgroup that exist
        const int pieces = (my_cols + 31) / 32;
        if (un.new_q) {
          __syncwarp();
          min_limit = INT_MAX;
          for (int c = lane; c < 64; c += 32) {
            const int f = un.rc * rows_per_chunk + wg * 64 + c;
            float nl = -INFINITY;
            int lim = -1;
            if (c < my_cols) {
              const int r = f / s.group;
              nl = -chain_load(lse + (long long)(un.row0 + r) * s.hq + un.g * s.group + f % s.group);
              if (lse_natural) nl = nl == nl && fabsf(nl) != INFINITY ? nl * kLog2e : -INFINITY;  // a row that sees no key adds 0
              lim = causal ? chain_load_cached(q_idx + un.row0 + r) : INT_MAX;
              min_limit = min(min_limit, lim);
            }
            neg_lse[c] = nl;
            limit[c] = lim;
          }
          min_limit = __reduce_min_sync(0xFFFFFFFFu, min_limit);
          __syncwarp();
        }
        float* out = partial + (long long)(un.g * rc_max + un.rc) * s.total_tokens + un.tok0;
        for (int t = 0; t < tiles; ++t, ++tile_no) {
          const int i = tile_no & 1;
          const uint32_t parity = (tile_no >> 1) & 1;
          ok = ptx::mbar_wait_warp(ptx::smem_u32(&ctl.tmem_full[i]), parity, abort);
          if (!ok) break;
          ptx::tc_fence_after_sync();
          const int key = key_begin + t * kTileKeys + my_lane;
          const bool masked = causal && (key_begin + t * kTileKeys + kTileKeys - 1 > min_limit);
          const uint32_t taddr = lane_addr + i * 256 + wg * 64;
          float sum = 0.f;
          if (pieces > 0)
            sum = masked ? sum_key_columns<true>(taddr, pieces, neg_lse, limit, key, s.scale_log2)
                         : sum_key_columns<false>(taddr, pieces, neg_lse, limit, key, s.scale_log2);
          if (wg > 0) {
            // sums[i] is free again: warpgroup 0 read it before it released accumulator i two tiles ago
            ctl.sums[i][wg - 1][my_lane] = sum;
            ptx::mbar_arrive(ptx::smem_u32(&ctl.sums_ready[i]));
          } else {
            ok = ptx::mbar_wait_warp(ptx::smem_u32(&ctl.sums_ready[i]), parity, abort);
            if (!ok) break;
#pragma unroll
            for (int w = 0; w < kGroups - 1; ++w) sum += ctl.sums[i][w][my_lane];
            if (key < un.n) out[key] = sum;
          }
          ptx::tc_fence_before_sync();
          ptx::mbar_arrive(ptx::smem_u32(&ctl.tmem_empty[i]));
        }
      }
    }
  }

  // ---- teardown: everybody meets here, whatever happened above ------------------------------------
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(tmem, kTmemCols);
  }
  if (threadIdx.x == 0 && ctl.abort && device_status) atomicOr(device_status, FASTAV_DEV_WAIT_EXPIRED);
}

// Fold the per-chunk (max, sum) pairs of a (scored row, head) into log2-sum-exp2.  Up to 32 pairs a row and 32 sequences: eight lanes per
// row, four pairs each in flight, and each lane of the warp knows where one sequence starts.  Else a warp per row, which looks its
// sequence up.  A call on 32 ragged sequences (28,672 rows) takes 295 us instead of 299 with a warp per row (the kernel took 9.2), on
// 4 x 16,384 tokens (16,384 rows of 30 pairs) 262 instead of 263.6; with two pairs kept the latter stay with the warp.
constexpr int kMergeKept = 4;
template <int LANES>
__global__ void __launch_bounds__(256) score_wide_merge_kernel(Shapes s, const int32_t* __restrict__ cu_qlens,
                                                               const int32_t* __restrict__ cu_seqlens,
                                                               const float2* __restrict__ stats, int stat_chunks,
                                                               int chunk_keys, float* __restrict__ lse) {
  chain_enter(s);
  pdl_wait();
  pdl_acquire(stats);
  pdl_acquire(cu_qlens);
  pdl_acquire(cu_seqlens);
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) / LANES, lane = threadIdx.x & 31, part = lane & (LANES - 1);
  const bool there = w < s.total_q * s.hq;
  if (LANES == 32 && !there) return;
  const int row = w / s.hq;
  int n = 0;
  if constexpr (LANES < 32) {
    const int b = min(lane, s.batch - 1), first = chain_load_cached(cu_qlens + b), count = seq_span<true>(s, cu_seqlens, b).count;
#pragma unroll
    for (int g = 0; g < 32 / LANES; ++g) {  // the last sequence that starts at or before the row of the warp's g-th entry
      const int wanted = __shfl_sync(0xFFFFFFFFu, row, g * LANES);
      const unsigned not_after = __ballot_sync(0xFFFFFFFFu, lane < s.batch && first <= wanted);
      const int found = __shfl_sync(0xFFFFFFFFu, count, not_after ? 31 - __clz(not_after) : 0);
      if (lane / LANES == g && not_after) n = found;
    }
  } else {
    // The row's sequence is the last one that starts at or before it.  The whole warp looks, 32 starts at a time: at evenly spaced
    // ones until at most 32 sequences are left, then at those (1,024 sequences: two rounds; one after the other 32 of them made a
    // score call of 1,024 x 128 tokens 169 us instead of 98).
    int lo = 0, left = s.batch;
    while (left > 32) {
      const int step = (left + 31) / 32, at = lo + lane * step;
      const unsigned not_after = __ballot_sync(0xFFFFFFFFu, lane * step < left && chain_load_cached(cu_qlens + at) <= row);
      const int skip = not_after ? (31 - __clz(not_after)) * step : 0;
      lo += skip;
      left = min(step, left - skip);
    }
    const int b = min(lo + lane, s.batch - 1);
    const int first = chain_load_cached(cu_qlens + b), count = seq_span<true>(s, cu_seqlens, b).count;
    const unsigned not_after = __ballot_sync(0xFFFFFFFFu, lane < left && first <= row);
    if (not_after) n = __shfl_sync(0xFFFFFFFFu, count, 31 - __clz(not_after));
  }
  const int chunks = there ? 2 * ((n + chunk_keys - 1) / chunk_keys) : 0;  // one entry per 64-key half of every tile run
  const float2* mine = stats + (long long)(there ? w : 0) * stat_chunks;
  // the first few entries of a lane stay in registers (usually all of them); the rest, if any, is read twice
  constexpr int kKept = LANES < 32 ? kMergeKept : 1;
  float2 kept[kKept];
#pragma unroll
  for (int u = 0; u < kKept; ++u) kept[u] = part + u * LANES < chunks ? chain_load(mine + part + u * LANES) : make_float2(-INFINITY, 0.f);
  float m = kept[0].x;
#pragma unroll
  for (int u = 1; u < kKept; ++u) m = fmaxf(m, kept[u].x);
  for (int t = part + kKept * LANES; t < chunks; t += LANES) m = fmaxf(m, chain_load(mine + t).x);
  __syncwarp();
#pragma unroll
  for (int d = LANES / 2; d; d >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
  float l = 0.f;
  if (m > -INFINITY) {
#pragma unroll
    for (int u = 0; u < kKept; ++u)
      if (kept[u].x > -INFINITY) l += kept[u].y * exp2f(kept[u].x - m);
    for (int t = part + kKept * LANES; t < chunks; t += LANES) {
      const float2 v = chain_load(mine + t);
      if (v.x > -INFINITY) l += v.y * exp2f(v.x - m);
    }
  }
  __syncwarp();
#pragma unroll
  for (int d = LANES / 2; d; d >>= 1) l += __shfl_xor_sync(0xFFFFFFFFu, l, d);
  if (part == 0 && there) lse[w] = (l > 0.f) ? m + log2f(l) : INFINITY;  // a row that sees no key contributes 0
}

constexpr int kFinalizeThreads = 64;

__global__ void __launch_bounds__(kFinalizeThreads) score_wide_finalize_kernel(Shapes s, const int32_t* __restrict__ cu_seqlens,
                                                                               const int32_t* __restrict__ cu_qlens, int rc_max,
                                                                               int rows_per_chunk, const float* __restrict__ partial,
                                                                               float* __restrict__ scores) {
  chain_enter(s);
  pdl_wait();
  pdl_acquire(partial);
  pdl_acquire(cu_seqlens);
  pdl_acquire(cu_qlens);
  const int b = blockIdx.y;
  const Span seq = seq_span<true>(s, cu_seqlens, b);
  const int tok0 = seq.first, n = seq.count;
  const int rows = row_span<true>(s, cu_qlens, b).count;
  const int row_chunks = (rows * s.group + rows_per_chunk - 1) / rows_per_chunk;
  const float inv = rows > 0 ? 1.0f / ((float)s.hq * (float)rows) : 0.f;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  scores[tok0 + j] = sum_of_partials<8>(partial + tok0 + j, s.hkv, row_chunks, rc_max, s.total_tokens) * inv;
}

// ---- host side -----------------------------------------------------------------------------------

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                   const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() { return reinterpret_cast<EncodeTiledFn>(tensor_map_encode_entry()); }

// Persistent grid and key chunk: one block per SM; chunks sized so that a block gets about seven units (fine
// enough to balance, and never more than its table holds).  Batches of so many sequences that no chunk does that take more
// blocks.
//
// Sequences of about one length (the longest at most a twentieth above the mean) are cut by what the busiest block has to do: it gets
// ceil(units / SMs) of them, 2,100 cycles per tile and 1,000 per unit (time stamps).  Seven units or so each are far from even where a
// remainder of the units takes a round of its own.  3 x 8,001-9,001 tokens, log-sum-exp given (chunks of 12 tiles instead of 2) 68.2 ->
// 66.8 us, 3 x 3,138-3,587, 109 rows (9 instead of 2) 63.8 -> 58.2.  Against seven units or so,
// measured on 140 drawn batches of this kind, heads of 64 and 128, with and without a given log-sum-exp: calls 3 % shorter on average, between
// 14 % and -1.6 %.  For ragged batches the mean says too little (the busiest block may get up to 45 % more, worked out).
long long busiest_block(long long groups, long long tiles, long long chunk_tiles) {
  const long long units = groups * ((tiles + chunk_tiles - 1) / chunk_tiles);
  return (units + kNumSMs - 1) / kNumSMs * ((tiles < chunk_tiles ? tiles : chunk_tiles) * 2100 + 1000);
}
long long even_chunk(const Shapes& s, int rc_max, long long chunk_tiles) {
  if (20ll * s.max_seqlen * s.batch > 21ll * s.total_tokens) return chunk_tiles;
  const long long groups = (long long)s.hkv * rc_max * s.batch, mean = s.total_tokens / s.batch, most = (s.max_seqlen + kTileKeys - 1) / kTileKeys;
  const long long fewer = mean < kTileKeys ? 1 : mean / kTileKeys, more = (s.total_tokens + (long long)s.batch * kTileKeys - 1) / ((long long)s.batch * kTileKeys);
  auto cost = [&](long long c) {  // whatever the sequences' lengths between these
    const long long a = busiest_block(groups, fewer, c), b = busiest_block(groups, more, c), d = busiest_block(groups, most, c);
    return a > b ? (a > d ? a : d) : (b > d ? b : d);
  };
  long long least = cost(chunk_tiles);
  for (int rounds = 1; rounds <= 12; ++rounds) {  // as many chunks per group as make that many units per block
    long long chunks = (long long)kNumSMs * rounds / groups;
    if (chunks < 1) continue;
    if (chunks > most) chunks = most;
    const long long c = (most + chunks - 1) / chunks, cycles = cost(c);
    if (cycles < least) {
      least = cycles;
      chunk_tiles = c;
    }
  }
  return chunk_tiles;
}
void plan_units(const Shapes& s, int rc_max, int* grid_out, int* chunk_tiles_out) {
  const long long tiles_upper = (long long)s.total_tokens / kTileKeys + s.batch;  // >= sum over sequences of ceil(n / 128)
  const long long tile_units = tiles_upper * s.hkv * rc_max;
  long long grid = tile_units < kNumSMs ? tile_units : kNumSMs;
  long long chunk_tiles = (tile_units + grid * kUnitsPerBlock - 1) / (grid * kUnitsPerBlock);
  if (chunk_tiles < 1) chunk_tiles = 1;
  chunk_tiles = even_chunk(s, rc_max, chunk_tiles);
  // units <= hkv * rc_max * (tokens / chunk + batch); keep the per-block share within the table
  auto units = [&] { return (long long)s.hkv * rc_max * (s.total_tokens / (chunk_tiles * kTileKeys) + s.batch); };
  while ((units() + grid - 1) / grid + 1 > kMaxUnits && chunk_tiles * kTileKeys <= s.total_tokens) ++chunk_tiles;
  if ((units() + grid - 1) / grid + 1 > kMaxUnits) grid = (units() + kMaxUnits - 2) / (kMaxUnits - 1);
  *grid_out = (int)grid;
  *chunk_tiles_out = (int)chunk_tiles;
}

template <int DIM>
cudaError_t run(const Shapes& s, const Workspace& w, const CUtensorMap& k_map, const CUtensorMap& q_map, const int32_t* q_idx,
                const int32_t* cu_qlens, const int32_t* cu_seqlens, const float* lse_in, float* scores_out, unsigned char* ws,
                int32_t* device_status, cudaStream_t stream, ScoreLeft* left) {
  float2* stats = reinterpret_cast<float2*>(ws + w.stats_off);
  float* lse = reinterpret_cast<float*>(ws + w.lse_off);
  float* partial = reinterpret_cast<float*>(ws + w.partial_off);
  // Partial sums per (KV head, chunk of query rows) -> scores: by the kernel that selects, or here.
  auto finish = [&](int row_chunks, int chunk) -> cudaError_t {
    if (left && (cluster_select_applies(s) || long_select_applies(s))) {
      left->kind = ScoreLeft::kPartials;
      left->row_chunks = row_chunks;
      left->rows_per_chunk = chunk;
      return cudaSuccess;
    }
    count_launches(1);
    return launch_chained(score_wide_finalize_kernel, dim3((s.max_seqlen + kFinalizeThreads - 1) / kFinalizeThreads, s.batch),
                          dim3(kFinalizeThreads), 0, stream, s, cu_seqlens, cu_qlens, row_chunks, chunk, (const float*)partial, scores_out);
  };
  OncePlan once;
  if (scores_out && (s.flags & FASTAV_SCORE_PATH_MASK) == 0 && once_plan(s, lse_in != nullptr, &once)) {
    const cudaError_t f = launch_score_once(s, &k_map, &q_map, q_idx, cu_qlens, cu_seqlens, lse_in, once, partial, device_status, stream);
    return f != cudaSuccess ? f : finish(once.row_tiles, once.rows_per_tile);
  }
  const int rows_per_chunk = wide_rows_per_chunk(s.group);
  const int rc_max = wide_row_chunks(s.max_qlen, s.group);
  int grid, chunk_tiles;
  plan_units(s, rc_max, &grid, &chunk_tiles);
  const int chunk_keys = chunk_tiles * kTileKeys;
  const int stat_chunks = 2 * ((s.max_seqlen + chunk_keys - 1) / chunk_keys);  // (max, sum) entries per (row, head)
  const int smem = Layout<DIM>::kTotal;
  cudaError_t e;
  e = once_per_context([&] {
    const cudaError_t f = cudaFuncSetAttribute(score_wide_kernel<DIM, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    return f == cudaSuccess ? cudaFuncSetAttribute(score_wide_kernel<DIM, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) : f;
  });
  if (e != cudaSuccess) return e;
  if (lse_in) {
    // The caller already has log-sum-exp per (row, head) (the layer's attention kernel returns it): one sweep.
    // Sweep 2 reads it as it is (an import kernel first: 3 x 8,001-9,001 tokens 69.7 us instead of 68.7).
  } else {
    if ((e = launch_chained(score_wide_kernel<DIM, 1>, dim3(grid), dim3(kThreads), smem, stream, k_map, q_map, s, q_idx, cu_qlens,
                            cu_seqlens, chunk_tiles, stat_chunks, rc_max, rows_per_chunk, stats, (const float*)nullptr,
                            0, (float*)nullptr, device_status)) != cudaSuccess)
      return e;
    const int entries = s.total_q * s.hq;
    const bool few_entries = s.batch <= 32 && stat_chunks <= 8 * kMergeKept;
    const auto merge = few_entries ? score_wide_merge_kernel<8> : score_wide_merge_kernel<32>;
    const int per_block = few_entries ? 32 : 8;
    if ((e = launch_chained(merge, dim3((entries + per_block - 1) / per_block), dim3(256), 0, stream, s, cu_qlens, cu_seqlens, (const float2*)stats,
                            stat_chunks, chunk_keys, lse)) != cudaSuccess)
      return e;
    count_launches(2);
  }
  if (!scores_out) return cudaGetLastError();  // only the statistics were asked for (fastav_lse)
  if ((e = launch_chained(score_wide_kernel<DIM, 2>, dim3(grid), dim3(kThreads), smem, stream, k_map, q_map, s, q_idx, cu_qlens,
                          cu_seqlens, chunk_tiles, stat_chunks, rc_max, rows_per_chunk, (float2*)nullptr,
                          lse_in ? lse_in : (const float*)lse, lse_in ? 1 : 0, partial, device_status)) != cudaSuccess)
    return e;
  count_launches(1);
  if ((e = finish(rc_max, rows_per_chunk)) != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace

void* tensor_map_encode_entry() {
  static void* entry = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult res;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &res) != cudaSuccess ||
        res != cudaDriverEntryPointSuccess)
      p = nullptr;
    return p;
  }();
  return entry;
}

bool encode_rows_map(const void* ptr, int dim, int heads, long long rows, long long st, long long sh, int box_heads, int box_rows,
                     void* map) {
  EncodeTiledFn encode = encode_tiled_fn();
  if (!encode || rows <= 0) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)dim, (cuuint64_t)heads, (cuuint64_t)rows};
  const cuuint64_t strides[2] = {(cuuint64_t)sh * 2, (cuuint64_t)st * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)box_heads, (cuuint32_t)box_rows};
  const cuuint32_t elem[3] = {1, 1, 1};
  return encode(static_cast<CUtensorMap*>(map), CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, elem,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Query rows per block: whole TMA boxes of 8 scored rows x G heads, as many as fit in 256 rows.
int wide_rows_per_chunk(int group) { return group >= 1 && group <= 32 ? kRowsPerCta / (8 * group) * (8 * group) : 0; }

int wide_row_chunks(int max_qlen, int group) {
  const int per = wide_rows_per_chunk(group);
  if (per == 0) return 1;
  const int c = (max_qlen * group + per - 1) / per;
  return c < 1 ? 1 : c;
}

bool score_wide_applies(const Shapes& s) {
  const auto ok_stride = [](long long v) { return v > 0 && v % 8 == 0 && (v >> 36) == 0; };
  return s.max_qlen >= 1 && s.total_q >= 1 && s.max_seqlen >= 1 && (s.dim == 64 || s.dim == 128) && s.group <= 32 &&
         ok_stride(s.k_st) && ok_stride(s.k_sh) && ok_stride(s.q_st) && ok_stride(s.q_sh);
}

cudaError_t launch_score_wide(const Shapes& s, const Workspace& w, const void* q, const int32_t* q_idx,
                              const int32_t* cu_qlens, const void* k, const int32_t* cu_seqlens, const float* lse_in,
                              float* scores_out, unsigned char* ws, int32_t* device_status, cudaStream_t stream, bool* used,
                              ScoreLeft* left) {
  CUtensorMap k_map, q_map;
  *used = encode_rows_map(k, s.dim, s.hkv, s.total_tokens, s.k_st, s.k_sh, 1, kTileKeys, &k_map) &&
          encode_rows_map(q, s.dim, s.hq, s.total_q, s.q_st, s.q_sh, s.group, 8, &q_map);
  if (!*used) return cudaSuccess;  // the caller falls back to the CUDA-core path
  if (s.dim == 128) return run<128>(s, w, k_map, q_map, q_idx, cu_qlens, cu_seqlens, lse_in, scores_out, ws, device_status, stream, left);
  return run<64>(s, w, k_map, q_map, q_idx, cu_qlens, cu_seqlens, lse_in, scores_out, ws, device_status, stream, left);
}

}  // namespace fastav
