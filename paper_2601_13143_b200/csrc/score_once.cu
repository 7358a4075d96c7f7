// Importance score, Eq. 4 (Section 2.2), for many scored rows on SHORT sequences: one pass over K.
//
// The long-sequence path (score_wide.cu) sweeps K twice because its logits fit nowhere.  Here they do: a thread-block cluster
// owns one tile of 128 query rows of one KV head, its blocks share out the keys, and a block's logits -- 128 rows x up to 512
// keys in fp32 -- stay in its 256 KB of tensor memory.  So
//
//   S = Q K^T per key tile (tcgen05.mma, operands by TMA), read once for the sum of 2^(z - top) per row and group of 32 keys, with the
//   2^(z - top) put back in its place; the blocks exchange the sums through distributed shared memory (one cluster barrier); each block
//   then adds its rows' sums up and reads again: 2^(z - top) 2^(top - lse), summed over the 128 rows of every key by a butterfly that
//   leaves one key per lane -> partial[KV head, row tile][token], which the selecting kernel (prune_few.cu, select_long.cu) adds up.
//   (With exponentials in both passes, prune of 1 x 2,048 tokens, 64 rows: 23.4 us instead of 22.6; the error against 64 bits is the same
//   on the whole, 0.6 to 1.8e-7 in the 2-norm.)  Where the caller hands the log-sum-exp in, S itself is read in the second pass.
//
// Two kernels (this and the selection) replace five (two sweeps, merge, per-token sums, selection).  Bound: latency, the
// chip is far from full.  Prune calls against the two-sweep path (28 / 4 heads, half the tokens kept): 32 rows on 1 x 1,024
// tokens 16.9 us instead of 28.9, 1 x 2,048 20.7 / 31.0, 4 x 2,048 36.3 / 50.1, 1 x 4,096 28.9 / 32.9; 128 rows on 1 x 2,048
// 25.9 / 37.7.
//
// A key's sums do not depend on its position (every column goes through the same arithmetic and the same tree), and a
// row's statistics are kept per key tile and folded in tile order, so that equal keys get bit-equal scores and a sequence's
// scores do not depend on the cluster's size.  All waits are bounded but the cluster's own barriers, which end because its blocks
// all run and every one of them arrives whatever happened before.
#include <cuda.h>
#include <limits.h>

#include "cluster.cuh"
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace fastav {
namespace {

constexpr int kTile = 128;                 // query rows of a tile; keys of a key tile
constexpr int kThreads = 576;              // warp 0: TMA, warp 1: MMA, warps 2-17: epilogue
constexpr int kEpilogueThreads = 512;
constexpr int kBlockTiles = 4;             // key tiles of a block: 512 columns of tensor memory
constexpr int kMaxTiles = kOnceMaxTokens / kTile;  // key tiles of a sequence
constexpr int kTmemCols = 512;
constexpr int kSubTileBytes = kTile * 128;

struct alignas(16) Control {
  uint64_t q_full, tmem_ready, k_full[kBlockTiles], s_full[kBlockTiles];
  uint32_t tmem_base;
  int abort;
  int index[4];
  int limit[kTile];                            // last key each row may see (-1: no such row)
  float neg_lse[kTile];
  float2 part[4][kBlockTiles][kTile];          // (top, sum of 2^(z - top)) per column group, key tile, row
  float2 run[4][kTile];                        // ... per run of the sequence's key tiles
  float2 fold[kTile];                          // per row: the second factor is 2^(top - x) y
  float2 stats[kMaxTiles][kTile];              // per key tile of the sequence: written by all blocks of the cluster
  float colsum[kBlockTiles][4][kTile];         // per key tile and 32-row quarter, the sums of every key
};

// Every block takes all of an SM's tensor memory, and the blocks of a cluster wait for one another: two clusters that met on
// two SMs could each hold one and want the other.  So no SM may hold two blocks, and what rules that out is shared memory
// (228 KB per SM, 1 KB of it per block not ours).
constexpr size_t kOneBlockBytes = 114 * 1024;
static_assert(2 * (kOneBlockBytes + 1024) > 228 * 1024, "two blocks would fit on an SM");
template <int DIM>
struct Layout {
  static constexpr int kOperandBytes = (DIM / 64) * kSubTileBytes;
  static constexpr size_t bytes(int tiles) {
    const size_t used = (size_t)(1 + tiles) * kOperandBytes + sizeof(Control) + 1024;
    return used > kOneBlockBytes ? used : kOneBlockBytes;
  }
};

__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kEpilogueThreads) : "memory"); }

// Lane j gets the sum over the warp's lanes of v[j]: at each step a lane gives away the half its partner keeps.
__device__ __forceinline__ float transpose_sum(float (&v)[32], int lane) {
#pragma unroll
  for (int half = 16; half >= 1; half >>= 1) {
    const bool upper = (lane & half) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float send = upper ? v[i] : v[i + half];
      const float keep = upper ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, send, half);
    }
  }
  return v[0];
}

// ---- 2^z in two factors ------------------------------------------------------------------------------
// The first pass leaves 2^(z - top) of every key, the second multiplies by 2^(top - lse).  `top` differs from one group of 32 keys to
// the next, and equal keys have to come out bit-equal all the same (with the group's own maximum taken off they differed by 1 to 3 units in the
// last place).  So nothing but a power of two is taken off: z = n + f, n the nearest integer and f rounded once, neither of which
// depends on `top`; 2^f has n - top added to its exponent; the row's factor is one over its sum with top - (the largest top) added; and
// their product is rounded once, to the same value wherever the key stands.  `top` is even, so that n is rounded the same way with it and
// without it, and above every z of its group, so that the first factor is at most 1.
//   Small values: the first factor stops at 2^-125, the second is at most 4 kLift, and their product is flushed below 2^-126: whichever
// factor would be too small, the key adds 0 in every group, as hidden keys do.  (kLift is undone in the partial sums.)
//   The integer's part costs 0.6 us of the 22.6 at 1 x 2,048 tokens.  Without it as long as all logits of a group are within 2^+-63, 22.1,
// but 24.2 to 26.2 where they are not, instead of 21.8 to 23.6.
constexpr float kLift = 0.0625f;
constexpr float kToInteger = 12582912.f;  // 1.5 x 2^23: the sum with it is rounded to an integer, which its low bits hold
constexpr float kMostTop = 65536.f;       // |top| up to which the kernel's own form is exact

__device__ __forceinline__ float top_of(float zmax) { return 2.f * floorf(0.5f * zmax) + 2.f; }

// 2^d of an integer d <= 127, 0 below 2^-126 and for NaN (the sum's low bits are d + 127).
__device__ __forceinline__ float power_of_two(float d) { return __int_as_float(__float_as_int(fmaxf(d, -127.f) + (kToInteger + 127.f)) << 23); }

// 2^(v * scale - top) for any v and any top above: NaN where the logit is not a number or +infinity.
__device__ __forceinline__ float exp_below(float v, float scale, float top) {
  const float z = v * scale;
  const bool exact = fabsf(z) < 4194304.f;  // (beyond, z is a multiple of 1/2)
  const float n = exact ? __fmaf_rn(v, scale, kToInteger) - kToInteger : rintf(z);
  const float f = exact ? __fmaf_rn(v, scale, -n) : z - n, d = n - top;
  const float p = d >= -125.f ? ptx::ex2_approx(f) * power_of_two(d) : 0.f;
  return z < INFINITY ? p : __int_as_float(0x7FFFFFFF);
}

// The first pass over a group of 32 keys where a row of the warp has logits that are far from 0, infinite or not a number: (top, sum).
// Rare, and short code rather than fast.
__device__ __forceinline__ float2 exponentials_far(uint32_t at, int bound, float scale) {
  float m = -INFINITY;  // (what is not a number is left out)
#pragma unroll 1
  for (int j0 = 0; j0 < 32; j0 += 8) {
    uint32_t v[8];
    ptx::tmem_ld8(at + j0, v);
    ptx::tmem_ld_wait_for(v);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j0 + j <= bound) m = fmaxf(m, __uint_as_float(v[j]));
  }
  const float top = m == -INFINITY ? 0.f : top_of(m * scale);
  float2 sum = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int j0 = 0; j0 < 32; j0 += 8) {
    uint32_t v[8];
    float p[8];
    ptx::tmem_ld8(at + j0, v);
    ptx::tmem_ld_wait_for(v);
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      p[j] = j0 + j <= bound ? exp_below(__uint_as_float(v[j]), scale, top) : 0.f;
      p[j + 1] = j0 + j + 1 <= bound ? exp_below(__uint_as_float(v[j + 1]), scale, top) : 0.f;
      sum = __fadd2_rn(sum, make_float2(p[j], p[j + 1]));
    }
    __syncwarp();
    ptx::tmem_st8(at + j0, p);
  }
  const float total = sum.x + sum.y;
  return make_float2(m == -INFINITY && total == total ? -INFINITY : top, total);
}

template <int DIM>
__global__ void __launch_bounds__(kThreads, 1)
score_once_kernel(const __grid_constant__ CUtensorMap k_map, const __grid_constant__ CUtensorMap q_map, Shapes s,
                  const int32_t* __restrict__ q_idx, const int32_t* __restrict__ cu_qlens, const int32_t* __restrict__ cu_seqlens,
                  const float* lse_in, int blocks, int rows_per_tile, int row_tiles, int tiles_per_block, float* __restrict__ partial,
                  int32_t* device_status) {
  using L = Layout<DIM>;
  constexpr int kSubTiles = DIM / 64;
  extern __shared__ unsigned char smem_raw[];
  cluster_arrive();  // "this block runs": waited for before the first remote access
  const uint32_t base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t q_smem = base, k_smem = base + L::kOperandBytes;
  Control& ctl = *reinterpret_cast<Control*>(smem_raw + (base - ptx::smem_u32(smem_raw)) + (1 + tiles_per_block) * L::kOperandBytes);
  volatile int* abort = &ctl.abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = (int)cluster_rank(), id = (int)blockIdx.x / blocks;
  const int rt = id % row_tiles, g = id / row_tiles % s.hkv, b = id / row_tiles / s.hkv;

  // Everything that touches no global memory comes before the wait of a call's first kernel.
  if (warp == 1) {
    if (lane == 0) {
      ptx::mbar_init(ptx::smem_u32(&ctl.q_full), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl.tmem_ready), 1);
      for (int i = 0; i < kBlockTiles; ++i) {
        ptx::mbar_init(ptx::smem_u32(&ctl.k_full[i]), 1);
        ptx::mbar_init(ptx::smem_u32(&ctl.s_full[i]), 1);
      }
      ctl.abort = 0;
      ptx::fence_barrier_init();
      ptx::prefetch_tensormap(&k_map);
      ptx::prefetch_tensormap(&q_map);
    }
  } else if (warp >= 2) {
    // The query tile starts as zeros: rows no copy ever fills are then harmless operands.
    for (int i = threadIdx.x - 64; i < L::kOperandBytes / 16; i += kEpilogueThreads)
      asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(q_smem + i * 16), "r"(0) : "memory");
    ptx::fence_proxy_async_smem();  // ordered before the TMA writes that follow the barrier
  }
  chain_enter_late(s, q_idx, cu_qlens, cu_seqlens);
  if (warp == 0) {  // the sequence's bounds, asked for by one warp
    const int32_t* word = lane < 2 ? cu_seqlens + b + lane : cu_qlens + b + (lane & 1);
    if (lane < 4) ctl.index[lane] = chain_load(word);
  }
  __syncthreads();
  const Span seq = checked_words(ctl.index[0], ctl.index[1], s.total_tokens, s.max_seqlen);
  const Span rows = checked_words(ctl.index[2], ctl.index[3], s.total_q, s.max_qlen);
  if (threadIdx.x == 0 && (seq.bad || rows.bad) && device_status) atomicOr(device_status, FASTAV_DEV_SHAPE_MISMATCH);
  const int n = min(seq.count, blocks * tiles_per_block * kTile);
  const int rows_here = min(rows_per_tile, rows.count * s.group - rt * rows_per_tile);  // of this row tile (a multiple of G)
  const int tiles = rows_here > 0 ? (n + kTile - 1) / kTile : 0;                         // key tiles of the sequence
  const int t0 = min(tiles, c * tiles_per_block);
  int mine = min(tiles - t0, tiles_per_block);
  const bool causal = (s.flags & FASTAV_CAUSAL) != 0;

  if (warp == 0) {
    pdl_wait();  // q and k may be what earlier work wrote
    if (mine > 0) {
      // Boxes of 8 scored rows x G heads x 64 columns land as 8 G consecutive 128-byte rows: the flat (scored row, head)
      // order of the tile, a whole number of 1024-byte swizzle groups.
      const int boxes = (rows_here / s.group + 7) / 8;
      const uint32_t box_bytes = 8u * s.group * 128u, bar = ptx::smem_u32(&ctl.q_full);
      ptx::mbar_expect_tx_warp(bar, boxes * box_bytes * kSubTiles);
      for (int i = 0; i < boxes; ++i)
#pragma unroll
        for (int sub = 0; sub < kSubTiles; ++sub)
          ptx::tma_load_3d_warp(q_smem + sub * kSubTileBytes + i * box_bytes, &q_map, sub * 64, g * s.group,
                                rows.first + rt * (rows_per_tile / s.group) + 8 * i, bar);
      for (int t = 0; t < mine; ++t) {
        const uint32_t k_bar = ptx::smem_u32(&ctl.k_full[t]);
        ptx::mbar_expect_tx_warp(k_bar, L::kOperandBytes);
#pragma unroll
        for (int sub = 0; sub < kSubTiles; ++sub)
          ptx::tma_load_3d_warp(k_smem + t * L::kOperandBytes + sub * kSubTileBytes, &k_map, sub * 64, g, seq.first + (t0 + t) * kTile, k_bar);
      }
      // The copies write into this block's shared memory: they have to be waited for before it may exit.
      int never = 0;
      ptx::mbar_wait_bounded(bar, 0, &never);
      for (int t = 0; t < mine; ++t) ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.k_full[t]), 0, &never);
    }
    __syncwarp();
  } else if (warp == 1) {
    // Tensor memory is taken when all earlier work has ended, never before: a block of an earlier kernel that starts its
    // successors first and allocates second would wait for this one's columns while this one waits for it.  The loads are on
    // their way meanwhile.
    pdl_wait();
    __syncwarp();
    ptx::tmem_alloc(ptx::smem_u32(&ctl.tmem_base), kTmemCols);
    ptx::tmem_relinquish();
    ptx::tc_fence_before_sync();
    ptx::mbar_arrive_warp(ptx::smem_u32(&ctl.tmem_ready), lane);
    const uint32_t tmem = ctl.tmem_base;
    // A wait that gives up changes nothing in the way the warp goes: see the epilogue.
    if (mine > 0) ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.q_full), 0, abort);
    for (int t = 0; t < mine; ++t) {
      ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.k_full[t]), 0, abort);
      ptx::tc_fence_after_sync();
      ptx::umma_bf16_steps<DIM / 16, kSubTileBytes, kSubTileBytes>(tmem + t * kTile, ptx::umma_desc_sw128(q_smem, 0),
                                                                   ptx::umma_desc_sw128(k_smem + t * L::kOperandBytes, 0),
                                                                   ptx::umma_idesc_bf16(kTile, kTile), false);
      ptx::umma_commit(ptx::smem_u32(&ctl.s_full[t]));
    }
    if (*abort && mine > 0) {  // the columns are given back below: not before the last MMA is done
      int never = 0;
      ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.s_full[mine - 1]), 0, &never);
    }
    __syncwarp();
  }
  const int quarter = warp & 3, cg = (warp - 2) >> 2;  // epilogue: TMEM lanes 32 quarter .., columns 32 cg .. of every key tile
  const int row_in = quarter * 32 + lane, ethread = cg * kTile + row_in;
  uint32_t lane_addr = 0;
  const float scale = s.scale_log2;
  const float2 sc = make_float2(scale, scale);
  const float inv_scale = 1.f / scale;
  bool ok = true;
  int limit = -1;
  if (warp >= 2) {
    pdl_wait();
    pdl_acquire(lse_in);
    if (cg == 0) {  // one column group asks, all four need it
      const int f = rt * rows_per_tile + row_in;
      int last = -1;
      float nl = -INFINITY;
      if (row_in < rows_here) {
        const int r = rows.first + f / s.group;
        last = min(n - 1, causal ? chain_load(q_idx + r) : INT_MAX);
        if (lse_in) {
          const float v = chain_load(lse_in + (long long)r * s.hq + g * s.group + f % s.group);
          nl = v == v && fabsf(v) != INFINITY ? -v * kLog2e : -INFINITY;  // a row that sees no key adds 0
        }
      }
      ctl.limit[row_in] = last;
      ctl.neg_lse[row_in] = nl;
    }
    epilogue_sync();
    limit = ctl.limit[row_in];
    // No tensor memory (one answer for the warp): nothing to read.  After that a wait that gives up only marks the results as
    // invalid: what follows it needs all lanes, so they all go on.
    const bool have_tmem = ptx::mbar_wait_warp(ptx::smem_u32(&ctl.tmem_ready), 0, abort);
    if (!have_tmem) mine = 0;
    ptx::tc_fence_after_sync();
    lane_addr = ctl.tmem_base + ((uint32_t)(quarter * 32) << 16) + cg * 32;
    pdl_trigger();
    if (!lse_in) {
      for (int t = 0; t < mine; ++t) {
        ok &= ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.s_full[t]), 0, abort);
        ptx::tc_fence_after_sync();
        uint32_t v[32];
        ptx::tmem_ld32(lane_addr + t * kTile, v);
        ptx::tmem_ld_wait_for(v);
        const int bound = limit - ((t0 + t) * kTile + cg * 32);  // columns 0..bound are visible
        if (bound < 31) {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (j > bound) v[j] = 0xFF800000u;  // -inf
        }
        float m0 = -INFINITY, m1 = -INFINITY;  // not a number if a logit is not
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          m0 = ptx::max_nan(m0, __uint_as_float(v[j]), __uint_as_float(v[j + 1]));
          m1 = ptx::max_nan(m1, __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
        }
        const float m = ptx::max_nan(m0, m1, -INFINITY), top = m == -INFINITY ? 0.f : top_of(m * scale), least = (top - 125.f) * inv_scale;
        if (__all_sync(0xFFFFFFFFu, m == -INFINITY || (fabsf(top) <= kMostTop && least < m))) {
          const float2 shift = make_float2(kToInteger - top, kToInteger - top);
          float2 sum = make_float2(0.f, 0.f);
          float p[32];
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            const float2 x = make_float2(fmaxf(__uint_as_float(v[j]), least), fmaxf(__uint_as_float(v[j + 1]), least));
            const float2 to = __ffma2_rn(x, sc, shift);                                          // kToInteger + n - top
            const float2 f = __ffma2_rn(x, sc, __ffma2_rn(to, make_float2(-1.f, -1.f), shift));  // z - n
            p[j] = __uint_as_float(__float_as_uint(ptx::ex2_approx(f.x)) + (__float_as_uint(to.x) << 23));
            p[j + 1] = __uint_as_float(__float_as_uint(ptx::ex2_approx(f.y)) + (__float_as_uint(to.y) << 23));
            sum = __fadd2_rn(sum, make_float2(p[j], p[j + 1]));
          }
          ctl.part[cg][t][row_in] = make_float2(m == -INFINITY ? -INFINITY : top, sum.x + sum.y);
          __syncwarp();  // rows differ in `bound`; the tcgen05 instructions need the whole warp
          ptx::tmem_st32(lane_addr + t * kTile, p);  // in place of the logits: the second pass needs no exponentials
        } else {
          ctl.part[cg][t][row_in] = exponentials_far(lane_addr + t * kTile, bound, scale);
        }
      }
    }
  }
  __syncwarp();
  cluster_wait();  // every block of the cluster runs
  if (!lse_in) {
    if (warp >= 2) {
      epilogue_sync();
      const int t = ethread >> 7, row = ethread & (kTile - 1);
      if (ok && t < mine) {  // one thread per (key tile, row): the four column groups, and off to every block
        float m = -INFINITY, l = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) m = fmaxf(m, ctl.part[i][t][row].x);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 p = ctl.part[i][t][row];
          l += p.y * power_of_two(p.x - m);
        }
        for (int q = 0; q < blocks; ++q) remote_store2(remote(&ctl.stats[t0 + t][row], q), __float_as_uint(m), __float_as_uint(l));
      }
    }
    cluster_sync();  // the last remote access
  }

  if (warp >= 2) {
    if (!lse_in) {
      // Each row's key tiles in four interleaved runs, in order, then the four.
      const int j = ethread >> 7, row = ethread & (kTile - 1);
      float m = -INFINITY, l = 0.f;
      for (int t = j; t < tiles; t += 4) m = fmaxf(m, ctl.stats[t][row].x);
      for (int t = j; t < tiles; t += 4) {
        const float2 p = ctl.stats[t][row];
        l += p.y * power_of_two(p.x - m);
      }
      ctl.run[j][row] = make_float2(m, l);
      epilogue_sync();
      if (ethread < kTile) {
        float mm = -INFINITY, total = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) mm = fmaxf(mm, ctl.run[i][ethread].x);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 p = ctl.run[i][ethread];
          total += p.y * power_of_two(p.x - mm);
        }
        ctl.fold[ethread] = make_float2(mm, total > 0.f && ethread < rows_here ? kLift * __frcp_rn(total) : 0.f);
      }
      epilogue_sync();
    }
    const float nl = ctl.neg_lse[row_in];
    const float2 nl2 = make_float2(nl, nl), fold = ctl.fold[row_in];
    __syncwarp();
    if (!lse_in) ptx::tmem_st_wait();
    for (int t = 0; t < mine; ++t) {
      if (lse_in) ok &= ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.s_full[t]), 0, abort);  // (else waited for above)
      ptx::tc_fence_after_sync();
      uint32_t v[32];
      ptx::tmem_ld32(lane_addr + t * kTile, v);
      ptx::tmem_ld_wait_for(v);
      float p[32];
      if (!lse_in) {
        const float w = fold.y * power_of_two(ctl.part[cg][t][row_in].x - fold.x);
#pragma unroll
        for (int j = 0; j < 32; ++j) p[j] = ptx::mul_ftz(__uint_as_float(v[j]), w);
      } else {
        const int bound = limit - ((t0 + t) * kTile + cg * 32);
#pragma unroll
        for (int j = 0; j < 32; j += 2) {
          const float2 z = __ffma2_rn(make_float2(__uint_as_float(v[j]), __uint_as_float(v[j + 1])), sc, nl2);
          p[j] = ptx::ex2_approx(z.x);
          p[j + 1] = ptx::ex2_approx(z.y);
        }
        if (bound < 31) {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (j > bound) p[j] = 0.f;
        }
      }
      __syncwarp();
      ctl.colsum[t][quarter][cg * 32 + lane] = transpose_sum(p, lane);
    }
    epilogue_sync();
    const int t = ethread >> 7, col = ethread & (kTile - 1), key = (t0 + t) * kTile + col;
    if (ok && t < mine && key < n)
      partial[(long long)(g * row_tiles + rt) * s.total_tokens + seq.first + key] =
          ((ctl.colsum[t][0][col] + ctl.colsum[t][1][col]) + (ctl.colsum[t][2][col] + ctl.colsum[t][3][col])) * (lse_in ? 1.f : 1.f / kLift);
  }

  // ---- teardown: everybody meets here, whatever happened above ------------------------------------
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(ctl.tmem_base, kTmemCols);
  }
  if (threadIdx.x == 0 && ctl.abort && device_status) atomicOr(device_status, FASTAV_DEV_WAIT_EXPIRED);
}

template <int DIM>
cudaError_t launch(const Shapes& s, const CUtensorMap& k_map, const CUtensorMap& q_map, const int32_t* q_idx, const int32_t* cu_qlens,
                   const int32_t* cu_seqlens, const float* lse_in, const OncePlan& plan, float* partial, int32_t* device_status, cudaStream_t stream) {
  const size_t smem = Layout<DIM>::bytes(plan.tiles_per_block);
  cudaError_t e = once_per_context([&] {
    cudaError_t f = cudaFuncSetAttribute(score_once_kernel<DIM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Layout<DIM>::bytes(kBlockTiles));
    if (f == cudaSuccess) f = cudaFuncSetAttribute(score_once_kernel<DIM>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return f;
  });
  if (e != cudaSuccess) return e;
  e = launch_chained_cluster(score_once_kernel<DIM>, dim3(s.batch * s.hkv * plan.row_tiles * plan.blocks), dim3(kThreads), plan.blocks, smem, stream,
                             k_map, q_map, s, q_idx, cu_qlens, cu_seqlens, lse_in, plan.blocks, plan.rows_per_tile, plan.row_tiles,
                             plan.tiles_per_block, partial, device_status);
  count_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// Query rows of a tile: whole TMA boxes of 8 scored rows x G heads (0: no box fits).
int once_rows_per_tile(int group) { return group >= 1 && group <= 16 ? kTile / (8 * group) * (8 * group) : 0; }
int once_row_tiles(int max_qlen, int group) {
  const int per = once_rows_per_tile(group);
  return per == 0 ? 0 : (max_qlen * group + per - 1) / per;
}

bool once_plan(const Shapes& s, bool lse_given, OncePlan* plan) {
  plan->rows_per_tile = once_rows_per_tile(s.group);
  if (plan->rows_per_tile == 0 || s.max_seqlen < 1 || s.max_qlen < 1) return false;
  plan->row_tiles = once_row_tiles(s.max_qlen, s.group);
  const int tiles = (s.max_seqlen + kTile - 1) / kTile;
  if (tiles > kMaxTiles) return false;
  const long long clusters = (long long)s.batch * s.hkv * plan->row_tiles;
  // Key tiles per block: the least time of all rounds (in quarters of a microsecond): a round of clusters that run at once takes
  // some 6 us and 3.75 us per key tile of a block (as fitted with exponentials in both passes; about 0.3 less since, so that a call near the
  // border may still go to the two sweeps where this would be a little quicker).  One round is always the better way (1 x 2,048 tokens, 32 rows, 28 / 4 heads:
  // 20.7 us with 2 key tiles per block in one round, 26.5 with 1 in two; the two sweeps 31.0).  Several rounds are compared with
  // the two sweeps: about 19 us, and per SM and key tile 2.25 us for every 128 rows of the first and 128 columns of the second.
  // Prune of 32 x 512 tokens, 32 rows: 60.0 against 71.1 us (32 / 8 heads: 66.8 against 83.4), 15 x 1,024: 57.9 / 64.5, but
  // 2 x 4,096 tokens, 32 / 8 heads: 57.9 / 52.8, 16 x 2,048, 8 rows, 32 / 8 heads: 127 / 116.
  long long least = LLONG_MAX;
  for (int per = 1; per <= kBlockTiles; ++per) {
    const int blocks = (tiles + per - 1) / per;
    if (blocks > s.cluster_limit) continue;
    const long long rounds = (clusters + kAtOnce[blocks] - 1) / kAtOnce[blocks], cost = rounds * (24 + 15 * per);
    if (cost >= least) continue;
    least = cost;
    plan->blocks = blocks;
    plan->tiles_per_block = per;
    plan->rounds = (int)(rounds < 100 ? rounds : 100);
  }
  if (least == LLONG_MAX) return false;
  if (plan->rounds == 1 || lse_given) return plan->rounds == 1;
  const long long key_tiles = s.total_tokens / kTile + (s.batch + 1) / 2;
  const int flat = s.max_qlen * s.group, chunk = wide_rows_per_chunk(s.group);
  long long per_tile = 0;  // of the first sweep in steps of 128 rows, of the second in rows
  for (int f = 0; f < flat; f += chunk) {
    const int rows = flat - f < chunk ? flat - f : chunk;
    per_tile += 9 * ((rows + 127) / 128) + 9 * (rows > 64 ? rows : 64) / 128;
  }
  const long long sweeps = 75 + key_tiles * s.hkv * per_tile / kNumSMs;
  return least + least / 32 < sweeps;
}

cudaError_t launch_score_once(const Shapes& s, const void* k_map, const void* q_map, const int32_t* q_idx, const int32_t* cu_qlens,
                              const int32_t* cu_seqlens, const float* lse_in, const OncePlan& plan, float* partial, int32_t* device_status,
                              cudaStream_t stream) {
  const CUtensorMap& km = *static_cast<const CUtensorMap*>(k_map);
  const CUtensorMap& qm = *static_cast<const CUtensorMap*>(q_map);
  return s.dim == 128 ? launch<128>(s, km, qm, q_idx, cu_qlens, cu_seqlens, lse_in, plan, partial, device_status, stream)
                      : launch<64>(s, km, qm, q_idx, cu_qlens, cu_seqlens, lse_in, plan, partial, device_status, stream);
}

}  // namespace fastav
