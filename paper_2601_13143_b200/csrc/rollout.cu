// Attention rollout (Section 2.1, "Analysis of audio-visual token importance via attention rollout", Eq. 2-3).
//
// Per layer: the head-mean attention map A^l of one sequence (tensor cores: S = Q_h K_h^T tile by tile, softmax
// weights from per-row log-sum-exp statistics that a first kernel computes or the caller hands in), Eq. 2
// (A~ = alpha A + (1 - alpha) I), and Eq. 3 as one n x n x n product R <- A~ R, again on the tensor cores.
//
// Precision.  The product runs in bf16 operands with fp32 accumulation, but both factors are kept as a PAIR of
// bf16 planes (x = hi + lo, hi = bf16(x), lo = bf16(x - hi): about 16 mantissa bits), and each product is the
// three leading terms hi*hi + lo*hi + hi*lo accumulated into the same TMEM tile, so that a chain of a dozen
// layers stays within about 1e-4 relative of the double-precision definition instead of drifting by 2^-9 per
// layer.
//
// Layout.  R is kept TRANSPOSED, RT[j][i] = R[i][j], row-major with the rows padded to n_pad = ceil(n / 128) *
// 128: then RT_new = RT_old * A~^T has both operands K-major (RT_old rows as the M side, A~ rows as the N
// side), which is what TMA tiles with the 128-byte swizzle feed to tcgen05.mma without any transpose.  Under
// the causal mask RT is upper and A~ lower triangular: RT's tiles below the diagonal stay the zeros that begin
// wrote, A~'s above it are neither written nor read, and the K loop of tile (m, n) only covers the blocks m..n.
//
// Sharing out the work.  At the paper's prompt size a layer is 171 visible 128 x 128 tiles on 148 SMs, so one block per tile
// and head, or per tile, leaves much of the chip idle in a second round, and the longest K loop of the triangular product
// alone is 36 blocks of 64.  The statistics kernel is PERSISTENT: its (head, row block, key block) items are cut into equal
// runs, one per SM, and a row block that several runs share leaves up to four partial log-sum-exps per row, which the map
// kernel merges when it reads them.  The map kernel cuts every row block into STRIPS of at most 32 .. 160 columns, the width
// that makes the fewest, fullest rounds.  The product cuts the K loops that are much longer than an SM's fair share into parts,
// whose fp32 tiles meet in the workspace: the part that finishes last adds them up in order (no block waits for another).
// 2,230 tokens, 28 / 4 heads of 128, per layer: statistics 34, map 37.4, product 21.1 us; 14 layers with their
// read-out 1,146 us (1,924 with a block per tile and head, or per tile).
//
// Warp 0 issues the TMA loads, warp 1 the MMAs into accumulators in tensor memory, warps 2..17 are the epilogue
// (thread <-> accumulator row, four warps per 32-lane quarter of TMEM, a quarter of the columns each).  The epilogue of
// the attention kernels is their bound: one exponential per element, 16 per clock and SM, and as much again of fixed cost per tile
// (a quarter of the exponentials on the FMA pipe instead: 0.5 to 1 %, and NaN came out as 2^-126).  All waits are bounded.  Where
// one gives up, the producer stops, and the warps that work together go on to the end of their lists on whatever there is, since what
// follows a wait there (elect.sync, tcgen05.ld, a warp's arrival) needs all lanes: every wait then returns after a few
// attempts, the results are marked invalid, and the way is the same for every lane.  (A vote per wait: 1,167 -> 1,186 us for 14
// layers of 2,230 tokens.)
#include <cuda.h>
#include <cuda_bf16.h>
#include <limits.h>
#include <math.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace fastav {
namespace {

constexpr int kTile = 128;
constexpr int kThreads = 576;
constexpr int kEpilogueThreads = 512;
constexpr int kColGroups = 4;  // epilogue warps per TMEM quarter; each takes 32 of the 128 columns
constexpr int kTmemCols = 512;
constexpr int kBuffers = 4;    // accumulators of 128 columns
constexpr int kMaxStripUnits = 5;  // the map's strips: up to 160 columns
constexpr int kMapBuffers = 3;     // accumulators of 160 columns
constexpr int kMaxStages = 4;
constexpr int kSubTileBytes = kTile * 128;  // 128 rows of one 64-element (128-byte) column block
constexpr int kMaxParts = 4;   // blocks that may share one row block's statistics
constexpr int kHeadChunk = 32;
constexpr size_t kPartialBytes = (size_t)kTile * kTile * sizeof(float);

template <int N>
struct IntTag {
  static constexpr int value = N;
};

struct alignas(16) PipeControl {
  uint64_t full[kMaxStages], empty[kMaxStages], tmem_full[kBuffers], tmem_empty[kBuffers], q_empty[2];
  uint32_t tmem_base;
  int abort;
  int last;                               // product: this block finished the tile's last part
};
struct AttnControl : PipeControl {
  union {
    float2 part[2][kColGroups - 1][kTile];  // statistics: (max, sum) per row of column groups 1..3
    float neg_lse[kHeadChunk][kTile];       // map: minus the log2-sum-exp2 of this strip's rows, some heads at a time
  };
};

__device__ __forceinline__ void split_bf16(float x, __nv_bfloat16& hi, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// A tile leaves through shared memory (the map's in the operand ring, which is idle by then): a thread holds columns of ONE row, and 32
// lanes that each store 16 bytes to another row fill half sectors of 32 rows at a time.  The accumulators are put down as
// they are, and a loop finishes 8 columns at a time, whole rows side by side.  Rows are an odd number of 16-byte pieces
// apart, so that the 8 rows of a quarter warp fall on different banks.  Product at 2,230 tokens: 28.3 -> 24.8 us.
constexpr int kStageStride = 32 * kMaxStripUnits + 4;  // floats
__device__ __forceinline__ void store_split(const float (&x)[8], __nv_bfloat16* hi, __nv_bfloat16* lo) {
  alignas(16) __nv_bfloat16 h[8], l[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) split_bf16(x[c], h[c], l[c]);
  *reinterpret_cast<uint4*>(hi) = *reinterpret_cast<const uint4*>(h);
  *reinterpret_cast<uint4*>(lo) = *reinterpret_cast<const uint4*>(l);
}
__device__ __forceinline__ void get8(const float* at, float (&x)[8]) {
  const float4 a = *reinterpret_cast<const float4*>(at), b = *reinterpret_cast<const float4*>(at + 4);
  x[0] = a.x, x[1] = a.y, x[2] = a.z, x[3] = a.w, x[4] = b.x, x[5] = b.y, x[6] = b.z, x[7] = b.w;
}

__device__ __forceinline__ float2 exp2_pair(float2 x) { return make_float2(ptx::ex2_approx(x.x), ptx::ex2_approx(x.y)); }

__device__ __forceinline__ void pipe_setup(PipeControl& ctl, int stages, int warp, const void* map_a, const void* map_b) {
  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; ++i) {
      ptx::mbar_init(ptx::smem_u32(&ctl.full[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl.empty[i]), 1);
    }
    for (int i = 0; i < kBuffers; ++i) {
      ptx::mbar_init(ptx::smem_u32(&ctl.tmem_full[i]), 1);
      ptx::mbar_init(ptx::smem_u32(&ctl.tmem_empty[i]), kEpilogueThreads / 32);
    }
    for (int i = 0; i < 2; ++i) ptx::mbar_init(ptx::smem_u32(&ctl.q_empty[i]), 1);
    ctl.abort = 0;
    ptx::fence_barrier_init();
    ptx::prefetch_tensormap(map_a);
    ptx::prefetch_tensormap(map_b);
  }
  if (warp == 1) {
    ptx::tmem_alloc(ptx::smem_u32(&ctl.tmem_base), kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before_sync();
  __syncthreads();
  ptx::tc_fence_after_sync();
}

__device__ __forceinline__ void pipe_teardown(PipeControl& ctl, int warp, int32_t* device_status) {
  ptx::tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc(ctl.tmem_base, kTmemCols);
  }
  if (threadIdx.x == 0 && ctl.abort && device_status) atomicOr(device_status, FASTAV_DEV_WAIT_EXPIRED);
}

// After giving up: copies already issued still write into this block's shared memory, so wait (bounded once
// more) for each of them before the block may exit.
__device__ __forceinline__ void drain_loads(PipeControl& ctl, int issued, int stages) {
  int never = 0;
  for (int t = max(0, issued - stages); t < issued; ++t)
    ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.full[t % stages]), (t / stages) & 1, &never);
}

// The MMAs a warp has issued still write tensor memory: the accumulator of the last of them, in turn with `buffers`, has to be
// done before the columns are given back.
__device__ __forceinline__ void drain_mmas(PipeControl& ctl, int issued, int buffers) {
  int never = 0;
  if (issued > 0) ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.tmem_full[(issued - 1) % buffers]), ((issued - 1) / buffers) & 1, &never);
  __syncwarp();
}

__device__ __forceinline__ void epilogue_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kEpilogueThreads) : "memory"); }

// ---- the flat list of items and its equal runs -------------------------------------------------------
__device__ __forceinline__ long long run_begin(long long items, int blocks, int b) { return items * b / blocks; }
// The block whose run holds item x.
__device__ __forceinline__ int run_of(long long items, int blocks, long long x) {
  int b = (int)((x * blocks) / items);
  while (run_begin(items, blocks, b + 1) <= x) ++b;
  while (run_begin(items, blocks, b) > x) --b;
  return b;
}
// Largest r with r (r + 1) / 2 <= x.
__device__ __forceinline__ int triangular_root(long long x) {
  int r = (int)((sqrtf(8.f * (float)x + 1.f) - 1.f) * 0.5f);
  while ((long long)(r + 1) * (r + 2) / 2 <= x) ++r;
  while ((long long)r * (r + 1) / 2 > x) --r;
  return r;
}

// ---- the attention map ---------------------------------------------------------------------------
// Shared memory of the statistics kernel: six tiles of 128 x DIM (192 KB at head_dim 128).
template <int DIM>
struct StatSmem {
  static constexpr int kSubTiles = DIM / 64;
  static constexpr int kOperandBytes = kSubTiles * kSubTileBytes;
  static constexpr int kStages = 4;  // the ring of K tiles; two more slots for Q tiles
  static constexpr size_t kBytes = (size_t)6 * kOperandBytes + sizeof(AttnControl) + 1024;
};

struct AttnArgs {
  int n, n_pad, hq, group;
  float scale_log2;
  int causal;
  float4* lse_parts;      // [hq][n_pad]: log2-sum-exp2 of up to four runs of a row's keys (-inf: no such run)
  int32_t* device_status;
};

// One item of the statistics: head, row block, key block, in that order.
struct StatItem {
  int head, rb, jb, blocks;
  bool causal;
  __device__ StatItem(long long x, int blocks_, bool causal_) : blocks(blocks_), causal(causal_) {
    const long long per_head = causal ? (long long)blocks * (blocks + 1) / 2 : (long long)blocks * blocks;
    head = (int)(x / per_head);
    const long long t = x % per_head;
    rb = causal ? triangular_root(t) : (int)(t / blocks);
    jb = (int)(t - (causal ? (long long)rb * (rb + 1) / 2 : (long long)rb * blocks));
  }
  __device__ __forceinline__ bool row_ends() const { return jb == (causal ? rb : blocks - 1); }
  __device__ __forceinline__ void advance() {
    if (!row_ends()) {
      ++jb;
      return;
    }
    jb = 0;
    if (++rb == blocks) {
      rb = 0;
      ++head;
    }
  }
};

// Per row and head, the log2-sum-exp2 of the scaled logits.
template <int DIM>
__global__ void __launch_bounds__(kThreads, 1)
rollout_stats_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map, AttnArgs a, long long items,
                     int* counters, int n_counters, ChainHead chain_head) {
  // The ring holds K tiles; a Q tile's slot is freed by the last MMA that reads it.
  using Cfg = StatSmem<DIM>;
  constexpr int kStages = Cfg::kStages, kOperandBytes = Cfg::kOperandBytes;
  extern __shared__ unsigned char smem_raw[];
  chain_enter_late(chain_head);
  const uint32_t base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t slots = base + kStages * kOperandBytes;
  AttnControl& ctl = *reinterpret_cast<AttnControl*>(smem_raw + (base - ptx::smem_u32(smem_raw)) + 6 * kOperandBytes);
  volatile int* abort = &ctl.abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int blocks = a.n_pad / kTile;
  const bool causal = a.causal != 0;
  const long long begin = run_begin(items, gridDim.x, blockIdx.x), end = run_begin(items, gridDim.x, blockIdx.x + 1);
  const int count = (int)(end - begin);

  pipe_setup(ctl, kStages, warp, &q_map, &k_map);
  const uint32_t tmem = ctl.tmem_base;

  if (warp == 0) {
    if (lane == 0) {
      pdl_wait();  // q and k may be what earlier work wrote
      StatItem x(begin, blocks, causal);
      int it = 0, loads = 0;  // items, Q tiles
      for (; it < count; ++it) {
        const int stage = it % kStages;
        if (!ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.empty[stage]), ((it / kStages) & 1) ^ 1u, abort)) break;
        const bool load_q = it == 0 || x.jb == 0;
        if (load_q && !ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.q_empty[loads & 1]), ((loads >> 1) & 1) ^ 1u, abort)) break;
        const uint32_t bar = ptx::smem_u32(&ctl.full[stage]);
        const uint32_t ring = base + stage * kOperandBytes, slot = slots + (loads & 1) * kOperandBytes;
        ptx::mbar_arrive_expect_tx(bar, kOperandBytes + (load_q ? kOperandBytes : 0));
#pragma unroll
        for (int sub = 0; sub < Cfg::kSubTiles; ++sub) {
          if (load_q) ptx::tma_load_3d(slot + sub * kSubTileBytes, &q_map, sub * 64, x.head, x.rb * kTile, bar);
          ptx::tma_load_3d(ring + sub * kSubTileBytes, &k_map, sub * 64, x.head / a.group, x.jb * kTile, bar);
        }
        loads += load_q;
        x.advance();
      }
      pdl_trigger();  // all loads have been issued
      if (*abort) drain_loads(ctl, it, kStages);
    }
  } else if (warp == 1) {
    {
      StatItem x(begin, blocks, causal);
      int loads = 0;
      for (int it = 0; it < count; ++it) {
        const int stage = it % kStages, buf = it % kBuffers;
        ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.full[stage]), (it / kStages) & 1, abort);
        ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.tmem_empty[buf]), ((it / kBuffers) & 1) ^ 1u, abort);
        ptx::tc_fence_after_sync();
        loads += it == 0 || x.jb == 0;
        const uint32_t k_tile = base + stage * kOperandBytes, q_tile = slots + ((loads - 1) & 1) * kOperandBytes;
        ptx::umma_bf16_steps<DIM / 16, kSubTileBytes, kSubTileBytes>(tmem + buf * kTile, ptx::umma_desc_sw128(q_tile, 0),
                                                                     ptx::umma_desc_sw128(k_tile, 0), ptx::umma_idesc_bf16(kTile, kTile), false);
        ptx::umma_commit(ptx::smem_u32(&ctl.empty[stage]));
        ptx::umma_commit(ptx::smem_u32(&ctl.tmem_full[buf]));
        if (x.row_ends()) ptx::umma_commit(ptx::smem_u32(&ctl.q_empty[(loads - 1) & 1]));
        x.advance();
      }
      if (*abort) drain_mmas(ctl, count, kBuffers);
    }
  } else {
    const int quarter = warp & 3, cg = (warp - 2) >> 2;  // TMEM lanes 32 quarter .., columns 32 cg ..
    const int row_in = quarter * 32 + lane, ethread = cg * kTile + row_in;
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16) + cg * 32;
    pdl_wait();
    for (int i = blockIdx.x * kEpilogueThreads + ethread; i < n_counters; i += gridDim.x * kEpilogueThreads) counters[i] = 0;
    StatItem x(begin, blocks, causal);
    // which of its row block's runs this block's first one is; every later row block starts here
    int part = blockIdx.x - run_of(items, gridDim.x, begin - x.jb);
    const float scale = a.scale_log2;
    const float2 sc = make_float2(scale, scale);
    float zmax = -INFINITY;  // unscaled
    float2 sum2 = make_float2(0.f, 0.f);
    int turn = 0;            // which half of the exchange buffer
    bool ok = true;
#pragma unroll 1
    for (int it = 0; it < count; ++it, x.advance()) {
      const int buf = it % kBuffers;
      ok &= ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.tmem_full[buf]), (it / kBuffers) & 1, abort);
      {
        ptx::tc_fence_after_sync();
        uint32_t v[32];
        ptx::tmem_ld32(lane_addr + buf * kTile, v);
        ptx::tmem_ld_wait_for(v);
        ptx::tc_fence_before_sync();
        ptx::mbar_arrive_warp(ptx::smem_u32(&ctl.tmem_empty[buf]), lane);  // the accumulator may be overwritten
        const int last_visible = min(a.n - 1, causal ? x.rb * kTile + row_in : INT_MAX);
        const int limit = last_visible - (x.jb * kTile + cg * 32);  // columns 0..limit of this group are visible
        if (limit < 31) {  // only tiles on the diagonal or at the end of the sequence
#pragma unroll
          for (int c = 0; c < 32; ++c)
            if (c > limit) v[c] = 0xFF800000u;  // -inf
        }
        if (limit >= 0) {
          float m = zmax;
#pragma unroll
          for (int c = 0; c < 32; c += 2) m = fmaxf(m, fmaxf(__uint_as_float(v[c]), __uint_as_float(v[c + 1])));
          const float corr = ptx::ex2_approx((zmax - m) * scale);  // 0 the first time
          sum2.x *= corr;
          sum2.y *= corr;
          zmax = m;
          const float shift = -m * scale;
          const float2 sh = make_float2(shift, shift);
#pragma unroll
          for (int c = 0; c < 32; c += 2)
            sum2 = __fadd2_rn(sum2, exp2_pair(__ffma2_rn(make_float2(__uint_as_float(v[c]), __uint_as_float(v[c + 1])), sc, sh)));
        }
        __syncwarp();  // the rows of a warp differ in `limit`; the tcgen05 instructions that follow need the whole warp
      }
      const bool row_ends = x.row_ends();
      if (!row_ends && it + 1 < count) continue;
      // the four column groups of a row meet in shared memory; group 0 writes the result
      if (cg > 0) ctl.part[turn][cg - 1][row_in] = make_float2(zmax, sum2.x + sum2.y);
      epilogue_sync();
      if (cg == 0 && ok) {
        float m = zmax;
#pragma unroll
        for (int g = 0; g < kColGroups - 1; ++g) m = fmaxf(m, ctl.part[turn][g][row_in].x);
        float total = zmax > -INFINITY ? (sum2.x + sum2.y) * ptx::ex2_approx((zmax - m) * scale) : 0.f;
#pragma unroll
        for (int g = 0; g < kColGroups - 1; ++g) {
          const float2 other = ctl.part[turn][g][row_in];
          if (other.x > -INFINITY) total += other.y * ptx::ex2_approx((other.x - m) * scale);
        }
        float* const out = reinterpret_cast<float*>(a.lse_parts + (long long)x.head * a.n_pad + x.rb * kTile + row_in);
        if (part < kMaxParts) out[part] = total > 0.f ? m * scale + log2f(total) : -INFINITY;
        if (row_ends)
          for (int p = part + 1; p < kMaxParts; ++p) out[p] = -INFINITY;
      }
      part = 0;
      turn ^= 1;
      zmax = -INFINITY;
      sum2 = make_float2(0.f, 0.f);
    }
  }
  pipe_teardown(ctl, warp, a.device_status);
}

// One block per strip: 128 rows of the map by 32 .. 160 of its columns.  `units` of 32 columns is the widest strip; a row block
// of U units that any row may see has ceil(U / units) strips of nearly equal width, long row blocks first.
struct MapStrip {
  int rb, unit, width;  // row block; first unit; units
  __device__ MapStrip(int t, int blocks, bool causal, int units) {
    for (rb = blocks - 1;; --rb) {
      const int all = 4 * (causal ? rb + 1 : blocks), strips = (all + units - 1) / units;
      if (t < strips || rb == 0) {
        unit = all * t / strips;
        width = all * (t + 1) / strips - unit;
        return;
      }
      t -= strips;
    }
  }
};

// Shared memory of the map kernel: a ring of Q tiles, one per head, and two slots for a strip of K, which is loaded once per
// KV head and shared by the G heads of its group (208 KB at head_dim 128).
template <int DIM>
struct MapSmem {
  static constexpr int kSubTiles = DIM / 64, kStages = 4, kSlots = 2;
  static constexpr int kOperandBytes = kSubTiles * kSubTileBytes;
  static constexpr int kStripSubBytes = 32 * kMaxStripUnits * 128;  // one 64-element column block of the widest strip
  static constexpr int kStripBytes = kSubTiles * kStripSubBytes;
  static constexpr size_t kBytes = (size_t)kStages * kOperandBytes + kSlots * kStripBytes + sizeof(AttnControl) + 1024;
  static_assert(kBytes <= 227 * 1024);
};

// Per strip: the sum over the heads of the softmax weights, then Eq. 2, stored as hi / lo planes (and, if asked, A itself in
// fp32).  Tiles no row may see, which the product never reads, are written only if the map is wanted.
template <int DIM>
__global__ void __launch_bounds__(kThreads, 1)
rollout_map_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_strip_map, AttnArgs a,
                   const float* __restrict__ lse_opt, float alpha, int units, int strips,
                   __nv_bfloat16* __restrict__ a_hi, __nv_bfloat16* __restrict__ a_lo, float* __restrict__ map_out, ChainHead chain_head) {
  using Cfg = MapSmem<DIM>;
  constexpr int kStages = Cfg::kStages, kOperandBytes = Cfg::kOperandBytes;
  constexpr int kStripCols = 32 * kMaxStripUnits;
  extern __shared__ unsigned char smem_raw[];
  chain_enter_late(chain_head);
  const uint32_t base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t slots = base + kStages * kOperandBytes;
  AttnControl& ctl =
      *reinterpret_cast<AttnControl*>(smem_raw + (base - ptx::smem_u32(smem_raw)) + kStages * kOperandBytes + Cfg::kSlots * Cfg::kStripBytes);
  volatile int* abort = &ctl.abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int blocks = a.n_pad / kTile, hq = a.hq, group = a.group;
  const bool causal = a.causal != 0;

  if ((int)blockIdx.x >= strips) {  // a tile no row may see, and the map is wanted: zeros (uniform for the block)
    pdl_wait();
    const int t = blockIdx.x - strips;                // (jb, rb) with jb > rb, in the order of the transposed triangle
    const int jb = triangular_root(t) + 1, rb = t - (jb - 1) * jb / 2;
    for (int i = threadIdx.x; i < kTile * kTile; i += kThreads) {
      const int r = rb * kTile + i / kTile, c = jb * kTile + i % kTile;
      if (r < a.n && c < a.n) map_out[(long long)r * a.n + c] = 0.f;
    }
    return;
  }
  const MapStrip strip(blockIdx.x, blocks, causal, units);
  const int rb = strip.rb;

  pipe_setup(ctl, kStages, warp, &q_map, &k_strip_map);
  const uint32_t tmem = ctl.tmem_base;

  if (warp == 0) {
    if (lane == 0) {
      pdl_wait();
      int it = 0;
      for (; it < hq; ++it) {
        const int stage = it % kStages;
        if (!ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.empty[stage]), ((it / kStages) & 1) ^ 1u, abort)) break;
        const uint32_t bar = ptx::smem_u32(&ctl.full[stage]);
        const bool load_k = it % group == 0;
        // the slot's last reader, two KV heads ago, if the wait above does not cover it
        const int reader = it - group - 1;
        if (load_k && reader >= 0 && reader > it - kStages &&
            !ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.empty[reader % kStages]), (reader / kStages) & 1, abort))
          break;
        const uint32_t ring = base + stage * kOperandBytes, slot = slots + ((it / group) & 1) * Cfg::kStripBytes;
        ptx::mbar_arrive_expect_tx(bar, kOperandBytes + (load_k ? Cfg::kSubTiles * strip.width * 4096 : 0));
#pragma unroll
        for (int sub = 0; sub < Cfg::kSubTiles; ++sub) {
          ptx::tma_load_3d(ring + sub * kSubTileBytes, &q_map, sub * 64, it, rb * kTile, bar);
          if (load_k)
            for (int u = 0; u < strip.width; ++u)
              ptx::tma_load_3d(slot + sub * Cfg::kStripSubBytes + u * 4096, &k_strip_map, sub * 64, it / group, (strip.unit + u) * 32, bar);
        }
      }
      pdl_trigger();  // all loads have been issued
      if (*abort) drain_loads(ctl, it, kStages);
    }
  } else if (warp == 1) {
    {
      const uint32_t idesc = ptx::umma_idesc_bf16(kTile, 32 * strip.width);
      for (int it = 0; it < hq; ++it) {
        const int stage = it % kStages, buf = it % kMapBuffers;
        ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.full[stage]), (it / kStages) & 1, abort);
        ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.tmem_empty[buf]), ((it / kMapBuffers) & 1) ^ 1u, abort);
        ptx::tc_fence_after_sync();
        const uint32_t q_tile = base + stage * kOperandBytes, k_tile = slots + ((it / group) & 1) * Cfg::kStripBytes;
        ptx::umma_bf16_steps<DIM / 16, kSubTileBytes, Cfg::kStripSubBytes>(tmem + buf * kStripCols, ptx::umma_desc_sw128(q_tile, 0),
                                                                           ptx::umma_desc_sw128(k_tile, 0), idesc, false);
        ptx::umma_commit(ptx::smem_u32(&ctl.empty[stage]));
        ptx::umma_commit(ptx::smem_u32(&ctl.tmem_full[buf]));
      }
      if (*abort) drain_mmas(ctl, hq, kMapBuffers);
    }
  } else {
    const int quarter = warp & 3, cg = (warp - 2) >> 2;  // TMEM lanes 32 quarter .., columns cols * cg ..
    const int row_in = quarter * 32 + lane, ethread = cg * kTile + row_in, row = rb * kTile + row_in;
    const int pieces = strip.width, cols = 8 * pieces;
    const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16) + cg * cols;
    pdl_wait();
    float4* lse_parts = a.lse_parts;
    pdl_acquire(lse_parts);
    pdl_acquire(lse_opt);
    const float2 sc = make_float2(a.scale_log2, a.scale_log2);
    // Statistics of the rows and heads from `it` on, `each` loads per thread in flight: one wait for
    // memory instead of eight (5,300 -> 3,100 cycles) where no accumulator needs the registers yet.
    auto stage_stats = [&](int it, auto each) {
      constexpr int kHeads = kEpilogueThreads / kTile, kEach = decltype(each)::value;
#pragma unroll 1
      for (int h0 = it + cg; h0 < min(it + kHeadChunk, hq); h0 += kEach * kHeads) {
        float4 st[kEach];
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
          const int h = h0 + i * kHeads;
          st[i] = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
          if (h < hq) {
            if (!lse_opt)
              st[i] = chain_load(lse_parts + (long long)h * a.n_pad + row);
            else if (row < a.n)
              st[i].x = chain_load(lse_opt + (long long)row * hq + h) * kLog2e;
          }
        }
#pragma unroll
        for (int i = 0; i < kEach; ++i) {
          float lse2 = st[i].x;
          if (st[i].y > -INFINITY) {  // several runs of the row's keys
            const float m = fmaxf(fmaxf(st[i].x, st[i].y), fmaxf(st[i].z, st[i].w));
            lse2 = m + log2f(ptx::ex2_approx(st[i].x - m) + ptx::ex2_approx(st[i].y - m) + ptx::ex2_approx(st[i].z - m) + ptx::ex2_approx(st[i].w - m));
          }
          ctl.neg_lse[h0 - it + i * kHeads][row_in] = fabsf(lse2) < INFINITY ? -lse2 : -INFINITY;  // a row that sees nothing adds 0
        }
      }
    };
    stage_stats(0, IntTag<8>{});
    epilogue_sync();
    float2 acc2[4 * kMaxStripUnits];
#pragma unroll
    for (int c = 0; c < 4 * kMaxStripUnits; ++c) acc2[c] = make_float2(0.f, 0.f);
    bool ok = true;
#pragma unroll 1
    for (int it = 0; it < hq; ++it) {
      const int buf = it % kMapBuffers;
      if (it > 0 && it % kHeadChunk == 0) {
        epilogue_sync();
        stage_stats(it, IntTag<1>{});
        epilogue_sync();
      }
      ok &= ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.tmem_full[buf]), (it / kMapBuffers) & 1, abort);
      ptx::tc_fence_after_sync();
      const float neg_lse2 = ctl.neg_lse[it % kHeadChunk][row_in];
      const float2 nl = make_float2(neg_lse2, neg_lse2);
      uint32_t v[32], v4[8];  // the fifth piece by itself
      const uint32_t from = lane_addr + buf * kStripCols;
      if (pieces >= 4) {
        ptx::tmem_ld32(from, v);
        if (pieces == 5) ptx::tmem_ld8(from + 32, v4);
      } else {
        ptx::tmem_ld8(from, v);
        if (pieces >= 2) ptx::tmem_ld8(from + 8, v + 8);
        if (pieces >= 3) ptx::tmem_ld8(from + 16, v + 16);
      }
      ptx::tmem_ld_wait_for(v, v4);
      ptx::tc_fence_before_sync();
      ptx::mbar_arrive_warp(ptx::smem_u32(&ctl.tmem_empty[buf]), lane);  // the accumulator may be overwritten
      auto weights = [&](const uint32_t* x) {
        return exp2_pair(__ffma2_rn(make_float2(__uint_as_float(x[0]), __uint_as_float(x[1])), sc, nl));
      };
      // Columns that a row may not see are added up too (a column's sum meets no other) and dropped when the tile is stored: with
      // two selects per pair the strips on the diagonal ended last (39.8 -> 37.4 us).
      if (pieces >= 4) {
#pragma unroll
        for (int c = 0; c < 32; c += 2) acc2[c / 2] = __fadd2_rn(acc2[c / 2], weights(v + c));
        if (pieces == 5) {
#pragma unroll
          for (int c = 0; c < 8; c += 2) acc2[16 + c / 2] = __fadd2_rn(acc2[16 + c / 2], weights(v4 + c));
        }
      } else {
#pragma unroll
        for (int p = 0; p < 3; ++p) {
          if (p < pieces) {
#pragma unroll
            for (int c = 8 * p; c < 8 * p + 8; c += 2) acc2[c / 2] = __fadd2_rn(acc2[c / 2], weights(v + c));
          }
        }
      }
    }
    float* const stage = reinterpret_cast<float*>(smem_raw + (base - ptx::smem_u32(smem_raw)));
    if (ok) {
      float* const at = stage + row_in * kStageStride + cg * cols;
#pragma unroll
      for (int c = 0; c < 4 * kMaxStripUnits; c += 2)
        if (2 * c < cols) *reinterpret_cast<float4*>(at + 2 * c) = make_float4(acc2[c].x, acc2[c].y, acc2[c + 1].x, acc2[c + 1].y);
    }
    epilogue_sync();
    if (ok) {
      const float inv_heads = 1.0f / (float)hq;
      const int chunks = 4 * pieces;  // of 8 columns
#pragma unroll 1
      for (int e = ethread; e < kTile * chunks; e += kEpilogueThreads) {
        const int r_in = e / chunks, c_in = (e - r_in * chunks) * 8;
        const int r = rb * kTile + r_in, col = strip.unit * 32 + c_in;
        const int last_visible = r < a.n ? min(a.n - 1, causal ? r : INT_MAX) : -1;
        float x[8];
        get8(stage + r_in * kStageStride + c_in, x);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float weight = col + c <= last_visible ? x[c] * inv_heads : 0.f;
          if (map_out && r < a.n && col + c < a.n) map_out[(long long)r * a.n + col + c] = weight;
          x[c] = alpha * weight + ((r < a.n && col + c == r) ? 1.0f - alpha : 0.f);  // Eq. 2
        }
        const long long at = (long long)r * a.n_pad + col;
        store_split(x, a_hi + at, a_lo + at);
      }
    }
  }
  pipe_teardown(ctl, warp, a.device_status);
}

// ---- Eq. 3: RT_new = RT_old * A~^T ------------------------------------------------------------------
// A unit is a part of a 128 x 128 tile of RT_new.  Per 64-wide K block the four operand tiles (RT hi, RT lo, A~ hi, A~ lo)
// are loaded once and used for the three products RT hi * A~ hi, RT lo * A~ hi, RT hi * A~ lo, all accumulated into the same
// TMEM tile.  Under the causal mask RT is upper and A~ lower triangular: tile (m, nn) has the K blocks m .. nn only, so
// that the tiles of one diagonal nn - m = d have 2 (d + 1) of them.  A tile is cut into ceil(its K blocks / share) equal
// parts; the parts are listed by decreasing d (the longest loops first, the short ones fill the tail), so the parts of
// cut tiles come first and a part's place in the workspace is its number.
// The kernel is persistent, one block per SM, and takes the list back and forth (block b: units b, 2 G - 1 - b, 2 G + b, ..):
// a unit's tile is stored while the next one's K loop runs on the other accumulator (24.8 -> 21.1 us at 2,230 tokens, with
// the limit of gemm_share; twelve MMAs of 64 cycles per K block are 6.2 us of it).
constexpr int kGemmStages = 3;
constexpr int kGemmStageBytes = 4 * kSubTileBytes;  // 128 x 64 each of RT hi, RT lo, A~ hi, A~ lo
constexpr int kGemmStageOut = 64 * kTile * sizeof(float);  // half a tile on its way out
struct GemmUnit {
  int mb, nb, kb0, kb1;  // tile; 64-wide K blocks [kb0, kb1)
  int part, parts;
  bool exists;
  __device__ GemmUnit(int u, int blocks, bool causal, int share) {
    exists = true;
    if (causal) {
      int d = blocks - 1;
      for (;; --d) {
        if (d < 0) {
          exists = false;
          return;
        }
        parts = (2 * (d + 1) + share - 1) / share;
        if (u < (blocks - d) * parts) break;
        u -= (blocks - d) * parts;
      }
      mb = u / parts;
      nb = mb + d;
    } else {
      parts = (2 * blocks + share - 1) / share;
      mb = u / parts / blocks;
      nb = u / parts % blocks;
      exists = mb < blocks;
    }
    part = u % parts;
    const int first = causal ? 2 * mb : 0, count = causal ? 2 * (nb - mb + 1) : 2 * blocks;
    kb0 = first + count * part / parts;
    kb1 = first + count * (part + 1) / parts;
  }
};

__global__ void __launch_bounds__(kThreads, 1)
rollout_gemm_kernel(const __grid_constant__ CUtensorMap rt_hi_map, const __grid_constant__ CUtensorMap rt_lo_map,
                    const __grid_constant__ CUtensorMap a_hi_map, const __grid_constant__ CUtensorMap a_lo_map, int n_pad,
                    int causal, int share, int units, __nv_bfloat16* __restrict__ out_hi, __nv_bfloat16* __restrict__ out_lo,
                    float* partials, int* counters, int32_t* device_status, ChainHead chain_head) {
  constexpr int kStages = kGemmStages, kStageBytes = kGemmStageBytes;
  extern __shared__ unsigned char smem_raw[];
  chain_enter_late(chain_head);
  const uint32_t base = (ptx::smem_u32(smem_raw) + 1023u) & ~1023u;
  PipeControl& ctl = *reinterpret_cast<PipeControl*>(smem_raw + (base - ptx::smem_u32(smem_raw)) + kStages * kStageBytes + kGemmStageOut);
  volatile int* abort = &ctl.abort;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int blocks = n_pad / kTile, grid = gridDim.x;
  auto unit_of = [&](int round) { return (round & 1) ? (round + 1) * grid - 1 - (int)blockIdx.x : round * grid + (int)blockIdx.x; };

  pipe_setup(ctl, kStages, warp, &rt_hi_map, &a_hi_map);
  const uint32_t tmem = ctl.tmem_base;

  if (warp == 0) {
    if (lane == 0) {
      pdl_wait();
      int it = 0;
      bool ok = true;
      for (int round = 0; ok && unit_of(round) < units; ++round) {
        const GemmUnit unit(unit_of(round), blocks, causal != 0, share);
        for (int kb = unit.kb0; kb < unit.kb1; ++kb, ++it) {
          const int stage = it % kStages;
          ok = ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.empty[stage]), ((it / kStages) & 1) ^ 1u, abort);
          if (!ok) break;
          const uint32_t bar = ptx::smem_u32(&ctl.full[stage]);
          const uint32_t dst = base + stage * kStageBytes;
          ptx::mbar_arrive_expect_tx(bar, kStageBytes);
          ptx::tma_load_2d(dst, &rt_hi_map, kb * 64, unit.mb * kTile, bar);
          ptx::tma_load_2d(dst + kSubTileBytes, &rt_lo_map, kb * 64, unit.mb * kTile, bar);
          ptx::tma_load_2d(dst + 2 * kSubTileBytes, &a_hi_map, kb * 64, unit.nb * kTile, bar);
          ptx::tma_load_2d(dst + 3 * kSubTileBytes, &a_lo_map, kb * 64, unit.nb * kTile, bar);
        }
      }
      pdl_trigger();  // all loads have been issued
      if (*abort) drain_loads(ctl, it, kStages);
    }
  } else if (warp == 1) {
    {
      int it = 0, round = 0;
      for (; unit_of(round) < units; ++round) {
        const GemmUnit unit(unit_of(round), blocks, causal != 0, share);
        const int buf = round & 1;
        ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.tmem_empty[buf]), ((round >> 1) & 1) ^ 1u, abort);
        for (int kb = unit.kb0; kb < unit.kb1; ++kb, ++it) {
          const int stage = it % kStages;
          ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.full[stage]), (it / kStages) & 1, abort);
          ptx::tc_fence_after_sync();
          const uint32_t rt_hi = base + stage * kStageBytes, rt_lo = rt_hi + kSubTileBytes, a_hi = rt_hi + 2 * kSubTileBytes,
                         a_lo = rt_hi + 3 * kSubTileBytes;
          const uint64_t rt_hi_desc = ptx::umma_desc_sw128(rt_hi, 0), rt_lo_desc = ptx::umma_desc_sw128(rt_lo, 0),
                         a_hi_desc = ptx::umma_desc_sw128(a_hi, 0), a_lo_desc = ptx::umma_desc_sw128(a_lo, 0);
          constexpr uint32_t idesc = ptx::umma_idesc_bf16(kTile, kTile);
          const uint32_t d = tmem + buf * kTile;
          ptx::umma_bf16_steps<4, 0, 0>(d, rt_hi_desc, a_hi_desc, idesc, kb > unit.kb0);
          ptx::umma_bf16_steps<4, 0, 0>(d, rt_lo_desc, a_hi_desc, idesc, true);
          ptx::umma_bf16_steps<4, 0, 0>(d, rt_hi_desc, a_lo_desc, idesc, true);
          ptx::umma_commit(ptx::smem_u32(&ctl.empty[stage]));
        }
        ptx::umma_commit(ptx::smem_u32(&ctl.tmem_full[buf]));
      }
      if (*abort) drain_mmas(ctl, round, 2);
    }
  } else {
    const int quarter = warp & 3, cg = (warp - 2) >> 2;
    const int row_in = quarter * 32 + lane, ethread = cg * kTile + row_in;
    pdl_wait();
    bool ok = true;
#pragma unroll 1
    for (int round = 0; unit_of(round) < units; ++round) {
      const int u = unit_of(round), buf = round & 1;
      const GemmUnit unit(u, blocks, causal != 0, share);
      ok &= ptx::mbar_wait_bounded(ptx::smem_u32(&ctl.tmem_full[buf]), (round >> 1) & 1, abort);
      float x[32];
      {
        ptx::tc_fence_after_sync();
        uint32_t v[32];
        ptx::tmem_ld32(tmem + ((uint32_t)(quarter * 32) << 16) + buf * kTile + cg * 32, v);
        ptx::tmem_ld_wait_for(v);
        ptx::tc_fence_before_sync();
        ptx::mbar_arrive_warp(ptx::smem_u32(&ctl.tmem_empty[buf]), lane);  // the accumulator may be overwritten
#pragma unroll
        for (int c = 0; c < 32; ++c) x[c] = __uint_as_float(v[c]);
      }
      bool mine = ok;  // this block writes the tile
      if (unit.parts > 1) {
        constexpr int kFloats = kTile * kTile;
        float* const here = partials + (size_t)u * kFloats + ethread;
#pragma unroll
        for (int c = 0; c < 32; ++c) __stcg(here + c * kEpilogueThreads, x[c]);
        __threadfence();
        epilogue_sync();
        if (ethread == 0) ctl.last = atomicAdd(counters + unit.mb * blocks + unit.nb, 1) == unit.parts - 1 && !ctl.abort;
        epilogue_sync();
        mine = ok && ctl.last != 0;
        if (mine) {  // the last part to finish: add the parts up in order
          __threadfence();
          const float* p = partials + (size_t)(u - unit.part) * kFloats + ethread;
#pragma unroll
          for (int c = 0; c < 32; ++c) x[c] = 0.f;
#pragma unroll 1
          for (int i = 0; i < unit.parts; ++i, p += kFloats) {
#pragma unroll
            for (int c = 0; c < 32; ++c) x[c] += __ldcg(p + c * kEpilogueThreads);
          }
        }
        if (!ctl.last) continue;  // (uniform for the epilogue)
      }
      // 64 rows at a time; a row's 16-byte pieces are permuted by its number, so that 8 rows fall on different banks
      float4* const stage = reinterpret_cast<float4*>(smem_raw + (base - ptx::smem_u32(smem_raw)) + kStages * kStageBytes);
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        if (quarter >> 1 == half) {
          const int r = row_in & 63;
#pragma unroll
          for (int c = 0; c < 32; c += 4)
            stage[r * 32 + ((cg * 8 + c / 4) ^ (r & 7))] = make_float4(x[c], x[c + 1], x[c + 2], x[c + 3]);
        }
        epilogue_sync();
        if (mine) {
#pragma unroll
          for (int i = 0; i < 64 * 16 / kEpilogueThreads; ++i) {
            const int e = ethread + i * kEpilogueThreads, r = e >> 4, c = e & 15;
            const float4 p = stage[r * 32 + ((2 * c) ^ (r & 7))], q = stage[r * 32 + ((2 * c + 1) ^ (r & 7))];
            const float y[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
            const long long at = (long long)(unit.mb * kTile + half * 64 + r) * n_pad + unit.nb * kTile + c * 8;
            store_split(y, out_hi + at, out_lo + at);
          }
        }
        epilogue_sync();
      }
    }
  }
  pipe_teardown(ctl, warp, device_status);
}

// ---- small kernels ----------------------------------------------------------------------------------
// RT <- I on the first n rows (the padding stays zero): 8 elements per thread.  The other copy's tiles below the diagonal become
// zeros: a causal layer writes none of them.
__global__ void rollout_identity_kernel(int n, int n_pad, __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                        __nv_bfloat16* __restrict__ other_hi, __nv_bfloat16* __restrict__ other_lo) {
  const long long i = ((long long)blockIdx.x * blockDim.x + threadIdx.x) * 8;
  if (i >= (long long)n_pad * n_pad) return;
  const int r = (int)(i / n_pad), c = (int)(i % n_pad);
  alignas(16) __nv_bfloat16 h[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) h[u] = __float2bfloat16_rn((r < n && c + u == r) ? 1.f : 0.f);
  *reinterpret_cast<uint4*>(hi + i) = *reinterpret_cast<const uint4*>(h);
  *reinterpret_cast<uint4*>(lo + i) = make_uint4(0, 0, 0, 0);
  if (r / kTile > c / kTile) {
    *reinterpret_cast<uint4*>(other_hi + i) = make_uint4(0, 0, 0, 0);
    *reinterpret_cast<uint4*>(other_lo + i) = make_uint4(0, 0, 0, 0);
  }
}

// importance[j] = (1 / n) sum_i R[i][j] = mean of row j of RT: one warp per row, a fixed summation order.
__global__ void __launch_bounds__(256) rollout_importance_kernel(int n, int n_pad, const __nv_bfloat16* __restrict__ hi,
                                                                  const __nv_bfloat16* __restrict__ lo,
                                                                  float* __restrict__ importance) {
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= n) return;
  const uint4 *h = reinterpret_cast<const uint4*>(hi + (long long)j * n_pad), *l = reinterpret_cast<const uint4*>(lo + (long long)j * n_pad);
  float total = 0.f;  // (the padding is zero)
#pragma unroll 4
  for (int i = lane; i < n_pad / 8; i += 32) {
    const uint4 x = h[i], y = l[i];
    const uint32_t hw[4] = {x.x, x.y, x.z, x.w}, lw[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int u = 0; u < 4; ++u)
      total += (__uint_as_float(hw[u] << 16) + __uint_as_float(lw[u] << 16)) + (__uint_as_float(hw[u] & 0xFFFF0000u) + __uint_as_float(lw[u] & 0xFFFF0000u));
  }
#pragma unroll
  for (int d = 16; d; d >>= 1) total += __shfl_xor_sync(0xFFFFFFFFu, total, d);
  if (lane == 0) importance[j] = total / (float)n;
}

// R[i][j] = RT[j][i] in fp32: 64 x 64 tiles through shared memory, read 8 elements at a time and written a row of 64 at a time
// (32 x 32 tiles with loads of 2 bytes kept too little in flight: 17.2 -> 8.7 us at 2,230 tokens; the whole read-out 16.4 ->
// 12.0 us, at 4,096 tokens 55.3 -> 33.3).
constexpr int kExportTile = 64;
__global__ void __launch_bounds__(256) rollout_export_kernel(int n, int n_pad, const __nv_bfloat16* __restrict__ hi,
                                                              const __nv_bfloat16* __restrict__ lo, float* __restrict__ out) {
  __shared__ float tile[kExportTile][kExportTile + 1];
  const int j0 = blockIdx.y * kExportTile, i0 = blockIdx.x * kExportTile;  // (n_pad is a multiple of 128: whole tiles exist)
#pragma unroll
  for (int e = threadIdx.x; e < kExportTile * kExportTile / 8; e += 256) {
    const int r = e / (kExportTile / 8), c = e % (kExportTile / 8) * 8;
    const long long at = (long long)(j0 + r) * n_pad + i0 + c;
    const uint4 x = *reinterpret_cast<const uint4*>(hi + at), y = *reinterpret_cast<const uint4*>(lo + at);
    const uint32_t hw[4] = {x.x, x.y, x.z, x.w}, lw[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      tile[r][c + 2 * u] = __uint_as_float(hw[u] << 16) + __uint_as_float(lw[u] << 16);
      tile[r][c + 2 * u + 1] = __uint_as_float(hw[u] & 0xFFFF0000u) + __uint_as_float(lw[u] & 0xFFFF0000u);
    }
  }
  __syncthreads();
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
#pragma unroll 4
  for (int r = ty; r < kExportTile; r += 8) {
    const int i = i0 + r;
    if (i >= n) break;
#pragma unroll
    for (int c = tx; c < kExportTile; c += 32)
      if (j0 + c < n) out[(long long)i * n + j0 + c] = tile[c][r];
  }
}

// keep mask and cut position from the importance: one block.
__global__ void __launch_bounds__(1024) rollout_threshold_kernel(int n, const float* __restrict__ importance, float threshold,
                                                                  const uint8_t* __restrict__ protect,
                                                                  uint8_t* __restrict__ keep_mask, int32_t* __restrict__ cut) {
  __shared__ int warp_last[32];
  int last = 0;  // one past the last unprotected token that reaches the threshold
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const bool reaches = importance[j] >= threshold, prot = protect && protect[j];
    keep_mask[j] = (reaches || prot) ? 1 : 0;
    if (reaches && !prot) last = j + 1;
  }
  last = __reduce_max_sync(0xFFFFFFFFu, last);
  if ((threadIdx.x & 31) == 0) warp_last[threadIdx.x >> 5] = last;
  __syncthreads();
  if (threadIdx.x < 32) {
    last = __reduce_max_sync(0xFFFFFFFFu, warp_last[threadIdx.x]);
    if (threadIdx.x == 0) *cut = last;
  }
}

// ---- host side ----------------------------------------------------------------------------------------
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                   const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                   CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// [n_pad, n_pad] bf16 row-major plane; a box is 128 rows of one 64-element column block.
bool plane_map(const void* ptr, int n_pad, CUtensorMap* map) {
  auto encode = reinterpret_cast<EncodeTiledFn>(tensor_map_encode_entry());
  if (!encode) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)n_pad, (cuuint64_t)n_pad};
  const cuuint64_t strides[1] = {(cuuint64_t)n_pad * 2};
  const cuuint32_t box[2] = {64, kTile};
  const cuuint32_t elem[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, elem,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// [tokens, heads, d] bf16 with element strides (st, sh, 1) as (d, heads, tokens); a box is 128 tokens, or `rows`, of one
// head's 64-element column block.  Tokens past the end read as zeros.
bool qk_map(const void* ptr, int dim, int heads, int tokens, long long st, long long sh, CUtensorMap* map, int rows = kTile) {
  auto encode = reinterpret_cast<EncodeTiledFn>(tensor_map_encode_entry());
  if (!encode) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)dim, (cuuint64_t)heads, (cuuint64_t)tokens};
  const cuuint64_t strides[2] = {(cuuint64_t)sh * 2, (cuuint64_t)st * 2};
  const cuuint32_t box[3] = {64, 1, (cuuint32_t)rows};
  const cuuint32_t elem[3] = {1, 1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, elem,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int pad_of(int n) { return (n + kTile - 1) / kTile * kTile; }
size_t plane_bytes(int n) { return (size_t)pad_of(n) * pad_of(n) * sizeof(__nv_bfloat16); }

// The state: copy 0 (hi, lo), copy 1 (hi, lo).
__nv_bfloat16* state_plane(void* state, int n, int copy, int lo) {
  return reinterpret_cast<__nv_bfloat16*>(static_cast<unsigned char*>(state) + (size_t)(copy * 2 + lo) * plane_bytes(n));
}

// ---- how a layer's work is shared out ------------------------------------------------------------------
long long visible_tiles(int blocks, bool causal) { return causal ? (long long)blocks * (blocks + 1) / 2 : (long long)blocks * blocks; }
long long hidden_tiles(int blocks) { return (long long)blocks * (blocks - 1) / 2; }

// Statistics: one run per SM unless the runs would get too short; a run of at least a third of the longest row block keeps
// the number of runs that share one within kMaxParts.
int stats_grid(int blocks, int hq, bool causal) {
  const long long g = visible_tiles(blocks, causal) * hq / ((blocks + 2) / 3);
  return (int)(g < 1 ? 1 : g > kNumSMs ? kNumSMs : g);
}

// Map: strips of at most `units` units of 32 columns.  Per head, a strip of u units takes some 350 + 270 u cycles (tiles of 128
// columns measured 1,430, strips of 160 1,700), and a block 6,000 before and after its heads; the width with the least
// rounds x cycles wins.  2,230 tokens, 28 heads: 144 strips of up to 160 columns are one round of 40.3 us, where 148 whole
// tiles and the other 23 in column slices of 32 were two of 51 us.
long long map_strips(int blocks, bool causal, int units) {
  long long strips = 0;
  for (int rb = 0; rb < blocks; ++rb) strips += (4 * (causal ? rb + 1 : blocks) + units - 1) / units;
  return strips;
}
int map_units(int blocks, bool causal, int hq) {
  int best = 1;
  long long least = LLONG_MAX;
  for (int units = 1; units <= kMaxStripUnits; ++units) {
    const long long rounds = (map_strips(blocks, causal, units) + kNumSMs - 1) / kNumSMs;
    const long long cycles = rounds * ((long long)hq * (350 + 270 * units) + 6000);
    if (cycles < least) {
      least = cycles;
      best = units;
    }
  }
  return best;
}

// Product: no K loop longer than one and a half times an SM's share of all K blocks, and at least twelve: a part costs an
// exchange of 64 KB, 4,000 to 8,000 cycles, the time of five to ten K blocks.  2,230 tokens (fair share 16): limits of
// 16 / 18 / 20 / 22 / 24 / 28 and none (36) took 23.9 / 23.0 / 22.1 / 21.1 / 21.1 / 22.3 / 25.6 us.
int gemm_share(int blocks, bool causal) {
  const long long items = causal ? (long long)blocks * (blocks + 1) * (blocks + 2) / 3 : 2ll * blocks * blocks * blocks;
  const long long share = (3 * items / 2 + kNumSMs - 1) / kNumSMs;
  return (int)(share < 12 ? 12 : share);
}
// Parts in all, and those of tiles that are cut (they come first).
void gemm_units(int blocks, bool causal, int share, int* units, int* cut) {
  *units = *cut = 0;
  for (int d = blocks - 1; d >= 0; --d) {
    const int count = causal ? 2 * (d + 1) : 2 * blocks, tiles = causal ? blocks - d : blocks, parts = (count + share - 1) / share;
    *units += tiles * parts;
    if (parts > 1) *cut += tiles * parts;
  }
}

struct RolloutWorkspace {
  size_t a_hi, a_lo, lse_parts, partials, counters, total;
  int n_counters;
};
RolloutWorkspace plan_rollout(int n, int hq) {
  RolloutWorkspace w{};
  const int blocks = pad_of(n) / kTile;
  int most = 0;  // parts that need a place, over both masks
  for (int causal = 0; causal < 2; ++causal) {
    int units, cut;
    gemm_units(blocks, causal != 0, gemm_share(blocks, causal != 0), &units, &cut);
    most = cut > most ? cut : most;
  }
  size_t off = 0;
  auto carve = [&](size_t bytes) { const size_t at = off; off = align_up(off + bytes, 256); return at; };
  w.a_hi = carve(plane_bytes(n));
  w.a_lo = carve(plane_bytes(n));
  w.lse_parts = carve((size_t)hq * pad_of(n) * sizeof(float4));
  w.partials = carve((size_t)most * kPartialBytes);
  w.n_counters = blocks * blocks;  // one per tile of the product
  w.counters = carve((size_t)w.n_counters * sizeof(int));
  w.total = off;
  return w;
}

template <int DIM>
cudaError_t run_attention(const fastav_params& p, const CUtensorMap& q_map, const CUtensorMap& k_map, const CUtensorMap& k_strip_map, const float* lse_opt, float alpha,
                          const RolloutWorkspace& w, unsigned char* ws, float* map_out, int32_t* device_status, cudaStream_t stream) {
  const bool causal = (p.flags & FASTAV_CAUSAL) != 0;
  const float scale = p.softmax_scale > 0.f ? p.softmax_scale : 1.0f / sqrtf((float)p.head_dim);
  AttnArgs a{};
  a.n = p.total_tokens;
  a.n_pad = pad_of(a.n);
  a.hq = p.num_q_heads;
  a.group = p.num_q_heads / p.num_kv_heads;
  a.scale_log2 = scale * kLog2e;
  a.causal = causal ? 1 : 0;
  a.lse_parts = reinterpret_cast<float4*>(ws + w.lse_parts);
  a.device_status = device_status;
  const int blocks = a.n_pad / kTile;
  int* counters = reinterpret_cast<int*>(ws + w.counters);
  cudaError_t e = once_per_context([&] {
    const cudaError_t f = cudaFuncSetAttribute(rollout_stats_kernel<DIM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)StatSmem<DIM>::kBytes);
    return f == cudaSuccess ? cudaFuncSetAttribute(rollout_map_kernel<DIM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MapSmem<DIM>::kBytes) : f;
  });
  if (e != cudaSuccess) return e;
  if (lse_opt) {
    e = cudaMemsetAsync(counters, 0, (size_t)w.n_counters * sizeof(int), stream);
  } else {
    e = launch_chained(rollout_stats_kernel<DIM>, dim3(stats_grid(blocks, a.hq, causal)), dim3(kThreads), StatSmem<DIM>::kBytes, stream, q_map, k_map, a,
                       visible_tiles(blocks, causal) * a.hq, counters, w.n_counters, ChainHead{});
    count_launches(1);
  }
  if (e != cudaSuccess) return e;
  const int units = map_units(blocks, causal, a.hq), strips = (int)map_strips(blocks, causal, units);
  const int zeros = map_out && causal ? (int)hidden_tiles(blocks) : 0;
  e = launch_chained(rollout_map_kernel<DIM>, dim3(strips + zeros), dim3(kThreads), MapSmem<DIM>::kBytes, stream, q_map, k_strip_map, a, lse_opt, alpha, units, strips,
                     reinterpret_cast<__nv_bfloat16*>(ws + w.a_hi), reinterpret_cast<__nv_bfloat16*>(ws + w.a_lo), map_out, ChainHead{});
  count_launches(1);
  return e;
}

bool aligned256(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 255u) == 0; }

}  // namespace
}  // namespace fastav

using namespace fastav;

extern "C" int32_t fastav_rollout_state_bytes(int32_t n, size_t* out_bytes) {
  if (!out_bytes || n < 1) return FASTAV_ERR_INVALID_ARG;
  if (n > FASTAV_ROLLOUT_MAX_TOKENS) return FASTAV_ERR_UNSUPPORTED;
  *out_bytes = 4 * plane_bytes(n);
  return FASTAV_OK;
}

extern "C" int32_t fastav_rollout_workspace_bytes(const fastav_params* p, size_t* out_bytes) {
  if (!p || !out_bytes || p->total_tokens < 1 || p->num_q_heads < 1) return FASTAV_ERR_INVALID_ARG;
  if (p->total_tokens > FASTAV_ROLLOUT_MAX_TOKENS) return FASTAV_ERR_UNSUPPORTED;
  *out_bytes = plan_rollout(p->total_tokens, p->num_q_heads).total;
  return FASTAV_OK;
}

extern "C" int32_t fastav_rollout_begin(int32_t n, void* state, size_t state_bytes, void* stream) {
  size_t need = 0;
  const int32_t rc = fastav_rollout_state_bytes(n, &need);
  if (rc != FASTAV_OK) return rc;
  if (!state || !aligned256(state) || state_bytes < need) return FASTAV_ERR_WORKSPACE;
  const int n_pad = pad_of(n);
  const long long threads = (long long)n_pad * n_pad / 8;
  rollout_identity_kernel<<<(unsigned)((threads + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      n, n_pad, state_plane(state, n, 0, 0), state_plane(state, n, 0, 1), state_plane(state, n, 1, 0), state_plane(state, n, 1, 1));
  count_launches(1);
  return cudaGetLastError() == cudaSuccess ? FASTAV_OK : FASTAV_ERR_CUDA;
}

extern "C" int32_t fastav_rollout_layer(const fastav_params* p, const void* q, const void* k, const float* lse_opt, float alpha,
                                        int32_t layer_index, void* state, size_t state_bytes, float* map_out_opt, void* workspace,
                                        size_t workspace_bytes, int32_t* device_status, void* stream) {
  if (!p || !q || !k || layer_index < 0 || !(alpha >= 0.f && alpha <= 1.f)) return FASTAV_ERR_INVALID_ARG;
  const int n = p->total_tokens;
  if (p->batch != 1 || n < 1 || p->total_q != n || p->max_seqlen != n || p->max_qlen != n) return FASTAV_ERR_INVALID_ARG;
  if (p->num_q_heads < 1 || p->num_kv_heads < 1 || p->num_q_heads % p->num_kv_heads != 0) return FASTAV_ERR_INVALID_ARG;
  if (p->head_dim != 64 && p->head_dim != 128) return FASTAV_ERR_UNSUPPORTED;
  if (n > FASTAV_ROLLOUT_MAX_TOKENS) return FASTAV_ERR_UNSUPPORTED;
  if (p->q_stride_head < p->head_dim || p->q_stride_tok < p->head_dim || p->k_stride_head < p->head_dim ||
      p->k_stride_tok < p->head_dim)
    return FASTAV_ERR_INVALID_ARG;
  if (p->q_stride_tok % 8 || p->q_stride_head % 8 || p->k_stride_tok % 8 || p->k_stride_head % 8 ||
      (reinterpret_cast<uintptr_t>(q) & 15u) || (reinterpret_cast<uintptr_t>(k) & 15u))
    return FASTAV_ERR_UNSUPPORTED;
  size_t need_state = 0, need_ws = 0;
  fastav_rollout_state_bytes(n, &need_state);
  fastav_rollout_workspace_bytes(p, &need_ws);
  if (!state || !aligned256(state) || state_bytes < need_state) return FASTAV_ERR_WORKSPACE;
  if (!workspace || !aligned256(workspace) || workspace_bytes < need_ws) return FASTAV_ERR_WORKSPACE;

  const int n_pad = pad_of(n);
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  const RolloutWorkspace w = plan_rollout(n, p->num_q_heads);
  const int src = layer_index & 1, dst = src ^ 1;
  CUtensorMap q_map, k_map, k_strip_map, rt_hi_map, rt_lo_map, a_hi_map, a_lo_map;
  if (!qk_map(q, p->head_dim, p->num_q_heads, n, p->q_stride_tok, p->q_stride_head, &q_map) ||
      !qk_map(k, p->head_dim, p->num_kv_heads, n, p->k_stride_tok, p->k_stride_head, &k_map) ||
      !qk_map(k, p->head_dim, p->num_kv_heads, n, p->k_stride_tok, p->k_stride_head, &k_strip_map, 32) ||
      !plane_map(state_plane(state, n, src, 0), n_pad, &rt_hi_map) || !plane_map(state_plane(state, n, src, 1), n_pad, &rt_lo_map) ||
      !plane_map(ws + w.a_hi, n_pad, &a_hi_map) || !plane_map(ws + w.a_lo, n_pad, &a_lo_map))
    return FASTAV_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  chain_begin(0);
  cudaError_t e = p->head_dim == 128 ? run_attention<128>(*p, q_map, k_map, k_strip_map, lse_opt, alpha, w, ws, map_out_opt, device_status, st)
                                     : run_attention<64>(*p, q_map, k_map, k_strip_map, lse_opt, alpha, w, ws, map_out_opt, device_status, st);
  if (e != cudaSuccess) return FASTAV_ERR_CUDA;
  constexpr size_t gemm_smem = kGemmStages * kGemmStageBytes + kGemmStageOut + sizeof(PipeControl) + 1024;
  static_assert(gemm_smem <= 227 * 1024);
  e = once_per_context([] { return cudaFuncSetAttribute(rollout_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem); });
  if (e != cudaSuccess) return FASTAV_ERR_CUDA;
  const bool causal = (p->flags & FASTAV_CAUSAL) != 0;
  const int blocks = n_pad / kTile, share = gemm_share(blocks, causal);
  int units, cut;
  gemm_units(blocks, causal, share, &units, &cut);
  const int grid = units < kNumSMs ? units : kNumSMs;
  e = launch_chained(rollout_gemm_kernel, dim3(grid), dim3(kThreads), gemm_smem, st, rt_hi_map, rt_lo_map, a_hi_map, a_lo_map, n_pad,
                     causal ? 1 : 0, share, units, state_plane(state, n, dst, 0), state_plane(state, n, dst, 1),
                     reinterpret_cast<float*>(ws + w.partials), reinterpret_cast<int*>(ws + w.counters), device_status, ChainHead{});
  count_launches(1);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? FASTAV_OK : FASTAV_ERR_CUDA;
}

extern "C" int32_t fastav_rollout_read(int32_t n, int32_t layers_applied, const void* state, size_t state_bytes,
                                       float* importance_out, float* rollout_out_opt, void* stream) {
  size_t need = 0;
  const int32_t rc = fastav_rollout_state_bytes(n, &need);
  if (rc != FASTAV_OK) return rc;
  if (layers_applied < 0 || !importance_out) return FASTAV_ERR_INVALID_ARG;
  if (!state || !aligned256(state) || state_bytes < need) return FASTAV_ERR_WORKSPACE;
  const int n_pad = pad_of(n), cur = layers_applied & 1;
  const __nv_bfloat16* hi = state_plane(const_cast<void*>(state), n, cur, 0);
  const __nv_bfloat16* lo = state_plane(const_cast<void*>(state), n, cur, 1);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  rollout_importance_kernel<<<(n + 7) / 8, 256, 0, st>>>(n, n_pad, hi, lo, importance_out);
  count_launches(1);
  if (rollout_out_opt) {
    const int tiles = (n + kExportTile - 1) / kExportTile;
    rollout_export_kernel<<<dim3(tiles, tiles), 256, 0, st>>>(n, n_pad, hi, lo, rollout_out_opt);
    count_launches(1);
  }
  return cudaGetLastError() == cudaSuccess ? FASTAV_OK : FASTAV_ERR_CUDA;
}

extern "C" int32_t fastav_rollout_threshold(int32_t n, const float* importance, float threshold, const uint8_t* protect_opt,
                                            uint8_t* keep_mask_out, int32_t* cut_out, void* stream) {
  if (n < 1 || !importance || !keep_mask_out || !cut_out) return FASTAV_ERR_INVALID_ARG;
  rollout_threshold_kernel<<<1, 1024, 0, static_cast<cudaStream_t>(stream)>>>(n, importance, threshold, protect_opt,
                                                                              keep_mask_out, cut_out);
  count_launches(1);
  return cudaGetLastError() == cudaSuccess ? FASTAV_OK : FASTAV_ERR_CUDA;
}
