// The kernel that selects: one thread-block CLUSTER per sequence goes from what scoring left to the keep list and (where that is
// little) the survivors' rows.
//
//   front   kKeys: few scored rows on a short sequence, nothing done yet -- the paper's own fine stage (Section 2.2, "Fine
//           pruning": one last-token query) on what the global stage left.  Q K^T by mma.sync, fragments loaded straight
//           from global memory (see KeyFragment); log-sum-exp per row and head (statistics per segment, exchanged through
//           distributed shared memory, one cluster barrier); then per token the fixed-order sum over heads and rows (Eq. 4).
//           kPartials: the tensor-core kernels' sums per (KV head, chunk of query rows) and token are added up.
//           kScores: finished scores (fastav_select).
//   select  the scores as order-preserving 32-bit keys (protected tokens: the largest) go to every block of the cluster, a
//           cluster barrier.  Up to 768 tokens (clusters of 16) each block then ranks its own slice by counting and tells the others how
//           many it keeps.  Beyond, each block runs the whole selection for itself: a histogram of the leading 12 bits,
//           the keys of the bin that holds the k-th largest finished by counting ranks (further 12-bit passes only if it holds
//           more than 256), one stable prefix sum in index order;
//   gather  the survivors among a block's own tokens.  From the keys, where shared memory holds the rows of its whole slice and at least half of
//           the call's tokens stay, they are on their way from the beginning and only stored at the end (512 tokens of a small model
//           10.1 -> 9.8 us, 4 stages from 563 tokens with rows of 1.5 KB 37.9 -> 35.5).
//
// Bound: latency.  Nothing here is long, so what counts is the number of dependent steps: every index array is asked for
// at once, the keys before anything that is only needed later, every reduction is spread over as many lanes as keep its
// order fixed, and nothing is computed by an owner that would have to publish it.  A prune call with one
// scored row (28 / 4 heads of 128, hidden 3,584, 80 % kept), this kernel and the compaction as they were first against the five kernels
// they stand for: 1 x 512 tokens 12.0 us instead of 20.7, 1 x 1,024 14.9 / 24.8, 1 x 2,048 18.3 / 28.8, 8 x 512 24.3 / 32.8.
//
// A sequence's scores depend on its length only, not on the cluster's size or the batch, and equal keys get bit-equal
// scores: all sums have a fixed order.
#include <math.h>

#include <atomic>

#include "cluster.cuh"
#include "common.cuh"
#include "gather.cuh"
#include "key_fragment.cuh"
#include "select_keys.cuh"
#include "sm100_ptx.cuh"

namespace fastav {
namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kPer = 4;                    // keys per thread in the selection
constexpr int kMaxTokens = kPer * kThreads;

enum Front { kKeys, kPartials, kScores };

constexpr int kDigitBits = 12;
constexpr int kBins = 1 << kDigitBits;
constexpr int kBinsPerThread = kBins / kThreads;
constexpr int kStatLanes = 8;   // lanes that share one (segment, term) of the row statistics
constexpr int kRowWarps = 8;    // warps that copy rows: the upper half, which short slices leave idle (all sixteen: 10.6 instead of 10.2 us for 512 tokens)
constexpr int kTokenLanes = 8;  // lanes that share one token's sum over the terms

// A sequence is cut into sixteen segments whatever the size of the cluster, and a block owns 16 / blocks of them: the row
// statistics are kept per segment and merged in a fixed tree.  Segments are whole fragments of 16 tokens (in steps of 32, 744 tokens
// kept twelve of sixteen blocks busy).
constexpr int kSegments = kMaxCluster;
__host__ __device__ inline int segment_of(int n) { return n <= 32 * kSegments ? 32 : ((n + kSegments - 1) / kSegments + 15) & ~15; }

struct FewArgs {
  const uint16_t* q;    // kKeys
  const uint16_t* k;
  const float* lse;     // kKeys, optional: the caller's natural-log log-sum-exp [total_q, Hq]
  int rq;               // kKeys: most scored rows of a sequence
  const float* in;      // kPartials [Hkv * row_chunks][N]; kScores [N]
  int row_chunks, rows_per_chunk;  // kPartials
  float* scores_out;    // [N] (not used by kScores)
  int do_select;        // 0: only the scores are wanted
  int do_gather;
  int early;            // the next kernel may start first thing
  int32_t* place;       // optional: see SelectArgs
  int ring;             // do_gather: where in shared memory the slice's rows are read to ahead of the selection; 0: they are not
  BulkPlan plan;        // ring
  int slice_cap;        // tokens per block that shared memory was sized for
  RowStreams rows;      // do_gather
};

// Short sequences are selected by counting: every block ranks its own slice's keys against all keys of the sequence, at most this
// many comparisons and tokens per block.  In place of five block-wide steps, one with no barrier inside and another exchange over the
// cluster; the comparisons grow with the square of the length.  From all keys to the keep list, by digits / by counting (time stamps):
// 512 tokens 2.3 / 1.9 us, 744 2.3 / 2.1, 820 2.4 / 2.9, 1,024 2.7 / 3.2 (by counting another 0.25 less from 513 to 768 since warps without
// tokens leave the comparisons out).
constexpr int kCountPairs = 36 << 10, kCountSlice = 256;

struct alignas(16) FewShared {
  unsigned hist[kBins];  // later: the block's survivors
  unsigned keys[kMaxTokens];
  unsigned prot_bits[kMaxTokens / 32];
  unsigned list[kDirectMax];
  int row_of[128], term_of[128];  // of a KV group's flat query row: scored row, term inside the group
  unsigned warp_a[kWarps];
  int limit[kNarrowMaxRows];
  int index[8];
  unsigned kept[kCountSlice / 32], kept_of[kMaxCluster];  // selection by counting: the block's survivors; how many each block has
  int base, list_n, remaining, bucket, need_eq, first_out, end_out, abort;
  unsigned prefix, threshold;
  uint64_t rows_full;  // the slice's rows have been read
};
static_assert(sizeof(FewShared) % 16 == 0 && kBins >= kMaxTokens, "what follows it stays 16-byte aligned");

// Dynamic shared memory after FewShared (bytes, every piece 16-byte aligned); host and device agree on it.
struct FewLayout {
  unsigned q, lse, stats, z, total;
};
__host__ __device__ inline int z_stride_of(int slice_cap) { return slice_cap + 4; }  // + 4: fragments store free of bank conflicts
__host__ __device__ inline FewLayout few_layout(int slice_cap, int terms, int dim) {
  FewLayout l{};
  unsigned at = 0;
  l.q = at;      // the query rows, 64 bytes of padding each
  at += (unsigned)terms * (dim * 2 + 64);
  l.lse = at;    // [terms]
  at += (unsigned)align_up((size_t)terms * 4, 16);
  l.stats = at;  // float2 [segments][terms], written by all blocks
  at += (unsigned)terms * kSegments * 8;
  l.z = at;      // [terms][z_stride]: this block's logits
  at += (unsigned)terms * z_stride_of(slice_cap) * 4;
  l.total = at;
  return l;
}

// The survivors' rows: not here, or copied from the keep list; not here, but every token's place is left; read ahead of the selection.
enum Rows { kByList, kPlaces, kAhead };

template <Front FRONT, int DIM, Rows ROWS>
__global__ void __launch_bounds__(kThreads, 1) prune_few_kernel(Shapes s, FewArgs a, const int32_t* __restrict__ cu_seqlens,
                                                                const int32_t* __restrict__ keep_counts,
                                                                const uint8_t* __restrict__ protect, const int32_t* __restrict__ q_idx,
                                                                const int32_t* __restrict__ cu_qlens, int32_t* __restrict__ keep_idx,
                                                                int32_t* __restrict__ cu_keep, int32_t* device_status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  FewShared& sh = *reinterpret_cast<FewShared*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int blocks = (int)gridDim.x / s.batch;  // blocks per cluster
  const int b = blockIdx.x / blocks, c = (int)cluster_rank();
  cluster_arrive();  // "this block runs": waited for before the first remote access

  // Whatever touches no global memory comes before the wait of a call's first kernel.
  const bool selecting = a.do_select != 0;
  if (selecting)
    for (int i = tid; i < kBins / 4; i += kThreads) reinterpret_cast<uint4*>(sh.hist)[i] = make_uint4(0, 0, 0, 0);
  if (tid < kMaxTokens / 32) sh.prot_bits[tid] = 0u;
  if (tid < kCountSlice / 32) sh.kept[tid] = 0u;
  if (tid == 32) {
    sh.base = 0;
    sh.list_n = 0;
  }
  if (ROWS == kAhead && tid == kThreads - 32) {
    sh.abort = 0;
    ptx::mbar_init(ptx::smem_u32(&sh.rows_full), 1);
    ptx::fence_barrier_init();
  }
  chain_enter_late(s, cu_seqlens, keep_counts, protect, q_idx, cu_qlens);
  if (a.early) pdl_trigger();  // (a second trigger below changes nothing)
  // ---- the caller's index arrays: one warp asks for all of them at once (sixteen warps of sixteen blocks asking for the
  //      same words queue at one L2 slice: 2,500 cycles instead of 900) ----------------------------------------------------
  if (warp == 0) {
    const int32_t* word = lane < 2 ? cu_seqlens + b + lane : lane < 4 ? cu_qlens + b + lane - 2 : keep_counts + b;
    // finished scores need the scored rows only where those survive by flag; without it the array may say anything
    const bool wants_rows = FRONT != kScores || (s.flags & FASTAV_PROTECT_QUERY_ROWS);
    const bool there = lane < 2 || (lane < 4 ? wants_rows : lane == 4 && selecting);
    const int v = there ? chain_load(word) : 0;
    if (lane < 5) sh.index[lane] = v;
  }
  __syncthreads();
  const Span seq = checked_words(sh.index[0], sh.index[1], s.total_tokens, s.max_seqlen);
  const Span qrows = checked_words(sh.index[2], sh.index[3], s.total_q, FRONT == kScores ? s.total_q : s.max_qlen);
  int k = sh.index[4];
  const bool k_clamped = k < 0 || k > seq.count;
  const int tok0 = seq.first, n = min(seq.count, a.slice_cap * blocks);
  const int seg = segment_of(n), slice = seg * (kSegments / blocks);  // tokens per segment, per block
  const int t0 = min(n, c * slice), m = min(n - t0, slice);           // this block's tokens: [t0, t0 + m) of the sequence
  const int all_rows = qrows.count, rows = min(all_rows, a.rq);
  const int flat = rows * s.group;  // query rows of one KV group, f = row * G + head of the group
  const int terms = s.hq * rows;    // term i = (head i / rows, row i % rows)
  const bool causal = (s.flags & FASTAV_CAUSAL) != 0;
  k = k < 0 ? 0 : (k > n ? n : k);

  // kKeys: the piece of the queries this thread stages first.
  constexpr int kQStride = DIM * 2 + 64;
  auto q_piece = [&](int i, int& at) -> const uint4* {  // piece i of the query rows; where it goes
    const int row = i / (DIM / 8), piece = i % (DIM / 8);  // row: (KV head, f)
    const int gg = row / flat, f = row - gg * flat, r = f / s.group;
    at = row * kQStride + piece * 16;
    return reinterpret_cast<const uint4*>(a.q + (long long)(qrows.first + r) * s.q_st + (long long)(gg * s.group + f - r * s.group) * s.q_sh + piece * 8);
  };
  const bool stages = FRONT == kKeys && tid < terms * (DIM / 8);
  int q_at = 0;
  const uint4* q_from = nullptr;
  if (stages) q_from = q_piece(tid, q_at);
  asm volatile("" : "+l"(q_from), "+r"(q_at));  // worked out ahead of the wait

  pdl_wait();
  // The scored rows' tokens survive (kKeys also needs them as the rows' limits).
  auto protect_rows = [&](int first_thread, int threads) {
    if (selecting && (s.flags & FASTAV_PROTECT_QUERY_ROWS))
      for (int r = tid - first_thread; r < all_rows; r += threads) {
        const int j = chain_load(q_idx + qrows.first + r) - t0;  // relative to this block's first token
        if (j >= 0 && j < m) atomicOr(&sh.prot_bits[j >> 5], 1u << (j & 31));
      }
  };
  // What the selection needs and nothing has needed so far.
  auto selection_inputs = [&] {
    if (!selecting) return;
    // output offset: the clamped keep counts of the sequences before this one, 32 per warp (up to 32 of them: the last warp)
    const int w = kWarps - 1 - warp;
    if (w * 32 < b) {
      int part = 0;
#pragma unroll 2
      for (int i = w * 32 + lane; i < b; i += kThreads) {
        const int ni = seq_span(s, cu_seqlens, i).count, ki = chain_load(keep_counts + i);
        part += ki < 0 ? 0 : min(ki, ni);
      }
      part = __reduce_add_sync(0xFFFFFFFFu, part);
      if (lane == 0 && part) atomicAdd(&sh.base, part);
    }
    if (protect)
      for (int j0 = warp * 32; j0 < m; j0 += kThreads) {  // a warp covers 32 tokens: one word
        const int j = j0 + lane;
        const unsigned word = __ballot_sync(0xFFFFFFFFu, j < m && chain_load(protect + tok0 + t0 + j) != 0);
        if (lane == 0 && word) atomicOr(&sh.prot_bits[j0 >> 5], word);
      }
    if (tid == 0 && c == 0 && k_clamped && device_status) atomicOr(device_status, FASTAV_DEV_K_CLAMPED);
  };
  // The slice's rows, survivors or not, into shared memory: half of the warps, a lane per piece of a row.
  Segment piece{};
  int pos_ahead = 0;
  const uint32_t ring = ptx::smem_u32(smem_raw) + a.ring, rows_bar = ptx::smem_u32(&sh.rows_full);
  bool copies = false;
  auto read_ahead = [&] {
    if (ROWS != kAhead) return;
    if (warp >= kWarps - kRowWarps) {
      copies = lane < a.plan.n_segments && make_segment(s, a.rows, lane, a.plan.packed_k, a.plan.packed_v, piece);
      if (tid == kThreads - 32 && m > 0) ptx::mbar_arrive_expect_tx(rows_bar, m * a.plan.row_bytes);
      for (int j = warp - (kWarps - kRowWarps); j < m; j += kRowWarps)
        if (copies) bulk_load(ring + j * a.plan.row_bytes + piece.slot_off, piece.in + (long long)(tok0 + t0 + j) * piece.in_stride, piece.bytes, rows_bar);
    }
    if (a.rows.pos_in && tid < m) pos_ahead = chain_load(a.rows.pos_in + tok0 + t0 + tid);
  };
  if (tid == 0 && (seq.bad || qrows.bad) && device_status) atomicOr(device_status, FASTAV_DEV_SHAPE_MISMATCH);
  const bool lowest = (s.flags & FASTAV_SELECT_LOWEST) != 0;
  auto key_of = [&](int j, float score) -> unsigned {  // token t0 + j of the sequence
    unsigned x = order_key(lowest ? -score : score);
    if (x == kProtectedKey) x = kProtectedKey - 1;  // only a NaN pattern lands here
    return ((sh.prot_bits[j >> 5] >> (j & 31)) & 1u) ? kProtectedKey : x;
  };
  if constexpr (FRONT == kKeys) {
    pdl_acquire(a.q);
    pdl_acquire(a.k);
    // ---- logits ----------------------------------------------------------------------------------------------
    const FewLayout lay = few_layout(a.slice_cap, s.hq * a.rq, DIM);
    unsigned char* const more = smem_raw + sizeof(FewShared);
    unsigned char* const q_sh = more + lay.q;
    float* const lse = reinterpret_cast<float*>(more + lay.lse);
    float2* const stats = reinterpret_cast<float2*>(more + lay.stats);
    float* const z = reinterpret_cast<float*>(more + lay.z);
    const int z_stride = z_stride_of(a.slice_cap);
    // Units of 16 tokens x one KV head, KV heads running fastest; the first one's keys are on their way before the queries
    // are staged.
    const int units = flat > 0 ? (m + 15) / 16 * s.hkv : 0;
    const uint16_t* const k_base = a.k + (long long)(tok0 + t0) * s.k_st;
    // Two fragments take turns: while one is multiplied the other is on its way.
    KeyFragment<DIM> even, odd;
    auto fetch = [&](KeyFragment<DIM>& frag, int u) {
      const int g = u % s.hkv, tok = u / s.hkv * 16;
      if (u < units) frag.load(k_base + (long long)tok * s.k_st + (long long)g * s.k_sh, s.k_st, m - tok, lane);
    };
    uint4 q_first = make_uint4(0, 0, 0, 0);
    if (stages) q_first = chain_load(q_from);  // the queries ahead of the keys: all warps wait for them together
    fetch(even, warp);
    fetch(odd, warp + kWarps);
    if (stages) *reinterpret_cast<uint4*>(q_sh + q_at) = q_first;
    for (int i = tid + kThreads; i < terms * (DIM / 8); i += kThreads) {
      int at;
      const uint4 v = chain_load(q_piece(i, at));
      *reinterpret_cast<uint4*>(q_sh + at) = v;
    }
    read_ahead();
    if (tid < flat) {
      sh.row_of[tid] = tid / s.group;
      sh.term_of[tid] = (tid % s.group) * rows + tid / s.group;
    }
    // what each scored row may see, relative to this block's first token (asked for beside the queries: both are one L2 latency)
    if (tid < kNarrowMaxRows) sh.limit[tid] = causal && tid < rows ? chain_load(q_idx + qrows.first + tid) - t0 : 0x7FFFFFFF;
    if (warp == 1) protect_rows(32, 32);
    __syncthreads();
    auto multiply = [&](const KeyFragment<DIM>& frag, int u) {
      const int g = u % s.hkv, j = u / s.hkv * 16 + (lane >> 2);
#pragma unroll 1
      for (int f0 = 0; f0 < flat; f0 += 8) {  // eight query rows at a time
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
        const unsigned char* const qp = q_sh + (g * flat + min(f0 + (lane >> 2), flat - 1)) * kQStride + (lane & 3) * 16;
#pragma unroll
        for (int i = 0; i < DIM / 32; ++i) {
          const uint4 qv = *reinterpret_cast<const uint4*>(qp + i * 64);
          mma_16x8x16(acc, frag.lo[i].x, frag.hi[i].x, frag.lo[i].y, frag.hi[i].y, qv.x, qv.y);
          mma_16x8x16(acc, frag.lo[i].z, frag.hi[i].z, frag.lo[i].w, frag.hi[i].w, qv.z, qv.w);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int f = f0 + (lane & 3) * 2 + e;
          if (f < flat) {
            const int lim = sh.limit[sh.row_of[f]];
            float* const at = z + (g * flat + sh.term_of[f]) * z_stride + j;
            at[0] = j <= lim ? acc[e] * s.scale_log2 : -INFINITY;
            at[8] = j + 8 <= lim ? acc[e + 2] * s.scale_log2 : -INFINITY;
          }
        }
        __syncwarp();
      }
    };
    for (int u = warp; u < units; u += 2 * kWarps) {
      multiply(even, u);
      fetch(even, u + 2 * kWarps);
      if (u + kWarps < units) multiply(odd, u + kWarps);
      fetch(odd, u + 3 * kWarps);
    }
    selection_inputs();  // arrives while other warps still multiply
    cluster_wait();
    __syncthreads();

    // ---- log-sum-exp per term ----------------------------------------------------------------------------------
    if (a.lse) {
      for (int i = tid; i < terms; i += kThreads) {
        const float v = chain_load(a.lse + (long long)(qrows.first + i % rows) * s.hq + i / rows);
        lse[i] = (v == v && fabsf(v) != INFINITY) ? v * kLog2e : INFINITY;  // a row that sees no key adds 0
      }
    } else {
      const int first_seg = t0 / seg, segs = (m + seg - 1) / seg, l8 = tid & (kStatLanes - 1);
#pragma unroll 1
      for (int i0 = 0; i0 < terms * segs; i0 += kThreads / kStatLanes) {  // (segment, term): running (max, sum 2^(z - max))
        const int i = i0 + tid / kStatLanes;
        const bool active = i < terms * segs;
        const int sg = segs == 1 ? 0 : i / terms, term = i - sg * terms, end = active ? min(m, (sg + 1) * seg) : 0;
        const float* const row = z + (active ? term : 0) * z_stride;
        float zm = -INFINITY, sum = 0.f;
#pragma unroll 1
        for (int j0 = sg * seg + l8; j0 < end; j0 += kStatLanes * 4) {
          float v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = j0 + kStatLanes * u < end ? row[j0 + kStatLanes * u] : -INFINITY;
          const float zn = fmaxf(zm, fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])));
          const float ref = zn == -INFINITY ? 0.f : zn;
          sum *= ptx::ex2_approx(zm - ref);
#pragma unroll
          for (int u = 0; u < 4; ++u) sum += ptx::ex2_approx(v[u] - ref);
          zm = zn;
        }
        __syncwarp();
        float bm = zm;
#pragma unroll
        for (int d = kStatLanes / 2; d; d >>= 1) bm = fmaxf(bm, __shfl_xor_sync(0xFFFFFFFFu, bm, d));
        sum = bm == -INFINITY ? 0.f : sum * ptx::ex2_approx(zm - bm);
#pragma unroll
        for (int d = kStatLanes / 2; d; d >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, d);
        if (active) {
          float2* const at = &stats[(first_seg + sg) * terms + term];
          for (int q = l8; q < blocks; q += kStatLanes) remote_store2(remote(at, q), __float_as_uint(bm), __float_as_uint(sum));
        }
      }
      cluster_sync();
      const int all_segs = (n + seg - 1) / seg, sg = tid & (kSegments - 1);
#pragma unroll 1
      for (int i0 = 0; i0 < terms; i0 += kThreads / kSegments) {  // a lane per segment
        const int i = i0 + tid / kSegments;
        float2 p = make_float2(-INFINITY, 0.f);
        if (i < terms && sg < all_segs) p = stats[sg * terms + i];
        float bm = p.x;
#pragma unroll
        for (int d = kSegments / 2; d; d >>= 1) bm = fmaxf(bm, __shfl_xor_sync(0xFFFFFFFFu, bm, d));
        float total = p.x > -INFINITY ? p.y * ptx::ex2_approx(p.x - bm) : 0.f;
#pragma unroll
        for (int d = kSegments / 2; d; d >>= 1) total += __shfl_xor_sync(0xFFFFFFFFu, total, d);
        if (i < terms && sg == 0) lse[i] = total > 0.f ? bm + __log2f(total) : INFINITY;
      }
    }
    __syncthreads();

    // ---- scores: eight lanes per token, each every eighth term in ascending order, added in a fixed tree ---------
    const float inv = all_rows > 0 ? 1.0f / ((float)s.hq * (float)all_rows) : 0.f;
    const int part = tid & (kTokenLanes - 1);
#pragma unroll 1
    for (int j0 = 0; j0 < m; j0 += kThreads / kTokenLanes) {
      const int j = j0 + tid / kTokenLanes;
      float total = 0.f;
      if (j < m) {
#pragma unroll 4
        for (int i = part; i < terms; i += kTokenLanes) total += ptx::ex2_approx(z[i * z_stride + j] - lse[i]);
      }
      __syncwarp();
#pragma unroll
      for (int d = kTokenLanes / 2; d; d >>= 1) total += __shfl_xor_sync(0xFFFFFFFFu, total, d);
      const float score = total * inv;
      if (j < m) {
        if (part == 0) a.scores_out[tok0 + t0 + j] = score;
        if (selecting) {
          const unsigned x = key_of(j, score);
          for (int q = part; q < blocks; q += kTokenLanes) remote_store(remote(&sh.keys[t0 + j], q), x);  // to every block of the cluster
        }
      }
    }
  } else {
    // ---- scores from partial sums, or as they are --------------------------------------------------------------------
    const float* in = a.in;
    pdl_acquire(in);
    protect_rows(0, kThreads);
    selection_inputs();
    cluster_wait();
    __syncthreads();
    const float* const col = in + tok0 + t0;
    if constexpr (FRONT == kPartials) {
      const int row_chunks = (all_rows * s.group + a.rows_per_chunk - 1) / a.rows_per_chunk;
      const float inv = all_rows > 0 ? 1.0f / ((float)s.hq * (float)all_rows) : 0.f;
      for (int j = tid; j < m; j += kThreads) {
        const float score = sum_of_partials<16>(col + j, s.hkv, row_chunks, a.row_chunks, s.total_tokens) * inv;
        a.scores_out[tok0 + t0 + j] = score;
        sh.keys[t0 + j] = key_of(j, score);
      }
    } else {
#pragma unroll 4
      for (int j = tid; j < m; j += kThreads) sh.keys[t0 + j] = key_of(j, chain_load(col + j));
    }
    __syncthreads();
    // This block's keys to everybody else, 16 bytes at a time (what lies past the last token is never read).
    const int quads = (m + 3) / 4;
    for (int q = 0; q < blocks; ++q) {
      if (q == c) continue;
      for (int i = tid; i < quads; i += kThreads) remote_store4(remote(&sh.keys[t0 + 4 * i], q), *reinterpret_cast<const uint4*>(&sh.keys[t0 + 4 * i]));
    }
  }
  if (!selecting) return;  // uniform for the cluster; nothing remote is outstanding
  int* const pos_sh = reinterpret_cast<int*>(smem_raw + a.ring + a.slice_cap * a.plan.row_bytes);
  if (ROWS == kAhead && tid < m) pos_sh[tid] = pos_ahead;
  if (ROWS == kPlaces) pdl_trigger();  // the gather reads its rows meanwhile: everything ahead of this kernel has ended
  cluster_sync();          // every block has all keys

  if (ROWS != kPlaces) pdl_trigger();
  const int base = sh.base;
  if (c == 0 && tid == 0) {
    cu_keep[b + 1] = base + k;
    if (b == 0) cu_keep[0] = 0;
    if (base + k > s.total_keep && device_status) atomicOr(device_status, FASTAV_DEV_SHAPE_MISMATCH);
  }
  const int room = s.total_keep - base;  // of the caller's keep list, from this sequence on
  auto rows_read = [&] {  // false: given up (one answer for the warp)
    if (m == 0 || ptx::mbar_wait_warp(rows_bar, 0, &sh.abort)) return true;
    if (lane == 0 && device_status) atomicOr(device_status, FASTAV_DEV_WAIT_EXPIRED);
    int never = 0;  // the copies in flight write into this block's shared memory: waited for once more, whichever warp gave up
    ptx::mbar_wait_bounded(rows_bar, 0, &never);
    return false;
  };
  if (k == 0) {  // nothing is kept, protected or not (uniform for the cluster)
    if (ROWS == kAhead) rows_read();  // (copies that write into this block's shared memory)
    if (ROWS == kPlaces)
      for (int j = tid; j < m; j += kThreads) a.place[tok0 + t0 + j] = -1;
    if (c == 0 && device_status)
      for (int j = tid; j < n; j += kThreads)
        if (sh.keys[j] == kProtectedKey) atomicOr(device_status, FASTAV_DEV_PROTECT_OVERFLOW);
    return;
  }
  const bool global_idx = (s.flags & FASTAV_KEEP_IDX_GLOBAL) != 0;
  unsigned* const picked = sh.hist;  // survivor `out` of the sequence is token picked[out % 4096]
  int first = 0, count = 0;          // this block's survivors

  if (slice <= kCountSlice && n * slice <= kCountPairs) {
    // ---- selection by counting (uniform for the cluster): some lanes per token of the slice, each compares it with every so
    //      many keys.  A token's rank is the number of keys above its own plus the equal ones of lower index. --------------
    const int tok_bits = slice <= 32 ? 1 : slice <= 64 ? 2 : slice <= 128 ? 3 : 4;  // tokens per warp; the lanes share them out
    const int j = (warp << tok_bits) + (lane & ((1 << tok_bits) - 1)), part = lane >> tok_bits, lanes = 32 >> tok_bits, at = t0 + j;
    const bool active = j < m;
    const unsigned own = active ? sh.keys[at] : 0xFFFFFFFFu;
    const uint4* const quads = reinterpret_cast<const uint4*>(sh.keys);
    int rank = 0;
    const int below = t0 / 4, slice_end = min((t0 + m + 3) / 4, n / 4), whole = n / 4;  // t0 is a multiple of 16
    int i = (warp << tok_bits) < m ? part : n;  // a warp without tokens has nothing to rank: whole blocks of them from 257 to 480 and 513 to 720 tokens
#pragma unroll 2
    for (; i < below; i += lanes) {  // tokens before the slice
      const uint4 v = quads[i];
      rank += (v.x >= own) + (v.y >= own) + (v.z >= own) + (v.w >= own);
    }
#pragma unroll 1
    for (; i < slice_end; i += lanes) {
      const uint4 v = quads[i];
      const int d = at - 4 * i;  // words 0 .. d - 1 come before the token
      rank += (v.x > own || (v.x == own && d > 0)) + (v.y > own || (v.y == own && d > 1)) + (v.z > own || (v.z == own && d > 2)) +
              (v.w > own || (v.w == own && d > 3));
    }
#pragma unroll 2
    for (; i < whole; i += lanes) {  // tokens behind it
      const uint4 v = quads[i];
      rank += (v.x > own) + (v.y > own) + (v.z > own) + (v.w > own);
    }
    for (i = n / 4 * 4 + part; i < n; i += lanes) rank += sh.keys[i] > own || (sh.keys[i] == own && i < at);  // the last few tokens
    __syncwarp();
    for (int d = 16; d >> tok_bits; d >>= 1) rank += __shfl_xor_sync(0xFFFFFFFFu, rank, d);
    const unsigned bits = __ballot_sync(0xFFFFFFFFu, part == 0 && active && rank < k);
    if (lane == 0 && bits) atomicOr(&sh.kept[(warp << tok_bits) >> 5], bits << ((warp << tok_bits) & 31));
    if (part == 0 && active && rank >= k && own == kProtectedKey && device_status)
      atomicOr(device_status, FASTAV_DEV_PROTECT_OVERFLOW);  // more protected tokens than k
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kCountSlice / 32; ++w) count += __popc(sh.kept[w]);
    if (tid < blocks) remote_store(remote(&sh.kept_of[c], tid), (unsigned)count);
    cluster_sync();  // the last remote access
    first = (int)__reduce_add_sync(0xFFFFFFFFu, lane < c ? sh.kept_of[lane] : 0u);
    const bool kept = tid < m && ((sh.kept[tid >> 5] >> lane) & 1u);
    if (tid < m && !kept && ROWS == kPlaces) a.place[tok0 + t0 + tid] = -1;
    if (kept) {
      int out = first + __popc(sh.kept[tid >> 5] & ((1u << lane) - 1u));
#pragma unroll
      for (int w = 0; w < kCountSlice / 32; ++w) out += w < (tid >> 5) ? __popc(sh.kept[w]) : 0;
      if (out < room) keep_idx[base + out] = (global_idx ? tok0 : 0) + t0 + tid;
      if (ROWS == kPlaces) a.place[tok0 + t0 + tid] = out < room ? base + out : -1;
      picked[out & (kBins - 1)] = (unsigned)(t0 + tid);
    }
  } else {
  // ---- selection by digits: thread t owns the tokens 4 t .. 4 t + 3 of the whole sequence ------------------------------
  const int mine = max(0, min(kPer, n - kPer * tid));
  unsigned x[kPer];
#pragma unroll
  for (int u = 0; u < kPer; u += 4) {
    const uint4 v = *reinterpret_cast<const uint4*>(&sh.keys[kPer * tid + u]);
    x[u] = v.x; x[u + 1] = v.y; x[u + 2] = v.z; x[u + 3] = v.w;
  }
  // The first pass looks at scores from 2^-63 up to 2 only, whose three leading bits are the same: a bin is 1/64 of an octave wide
  // instead of 1/8, and the bin of the k-th largest holds few keys to rank.  Smaller scores share the lowest bin, larger ones (and
  // protected tokens) the highest; where the k-th largest lies in one of these two among many, the passes start again from the first bit.
  // (From the keys only: three stages from 1,024 tokens 36.6 -> 36.3 us; from partial sums 1 x 2,048 tokens 21.5 -> 21.6.)
  constexpr int kWindowShift = 29 - kDigitBits;
  const int window = lowest ? 2 << kDigitBits : 5 << kDigitBits;
  auto window_digit = [&](unsigned key) { return (unsigned)min(max((int)(key >> kWindowShift) - window, 0), kBins - 1); };
  bool windowed = FRONT == kKeys;
  unsigned prefix = 0u;   // the bits of the k-th largest key fixed so far
  int remaining = k, bits_left = 32;
#pragma unroll 1
  for (int pass = 0; bits_left > 0; ++pass) {
    const int shift = windowed ? kWindowShift : max(0, bits_left - kDigitBits);
    const unsigned above_want = __funnelshift_rc(prefix, 0u, bits_left);  // prefix >> bits_left, 0 for 32
    if (pass > 0) {
      for (int i = tid; i < kBins / 4; i += kThreads) reinterpret_cast<uint4*>(sh.hist)[i] = make_uint4(0, 0, 0, 0);
      __syncthreads();
    }
    {
      unsigned run_digit = kBins, run_len = 0u;  // equal digits of consecutive tokens (typically zeros): one update
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        if (u < mine && __funnelshift_rc(x[u], 0u, bits_left) == above_want) {
          const unsigned digit = windowed ? window_digit(x[u]) : (x[u] >> shift) & (kBins - 1);
          if (digit != run_digit) {
            if (run_len) atomicAdd(&sh.hist[run_digit], run_len);
            run_digit = digit;
            run_len = 0u;
          }
          ++run_len;
        }
      }
      if (run_len) atomicAdd(&sh.hist[run_digit], run_len);
    }
    __syncthreads();
    unsigned h[kBinsPerThread], own = 0;
#pragma unroll
    for (int i = 0; i < kBinsPerThread; i += 4) {
      const uint4 v = *reinterpret_cast<const uint4*>(&sh.hist[tid * kBinsPerThread + i]);
      h[i] = v.x; h[i + 1] = v.y; h[i + 2] = v.z; h[i + 3] = v.w;
      own += v.x + v.y + v.z + v.w;
    }
    unsigned above = sum_above<kWarps>(own, sh.warp_a, lane, warp);
    const unsigned rem = (unsigned)remaining;
    if (above < rem && rem <= above + own) {  // exactly one thread: its bins from the top
#pragma unroll
      for (int i = kBinsPerThread - 1; i >= 0; --i) {
        if (above < rem && rem <= above + h[i]) {
          sh.prefix = windowed ? (unsigned)(tid * kBinsPerThread + i) : prefix | ((unsigned)(tid * kBinsPerThread + i) << shift);
          sh.remaining = (int)(rem - above);
          sh.bucket = (int)h[i];
        }
        above += h[i];
      }
    }
    __syncthreads();
    const unsigned found = sh.prefix;
    const bool in_window = windowed;
    if (windowed) {
      windowed = false;
      if ((found == 0u || found == kBins - 1) && sh.bucket > kDirectMax) continue;  // (prefix and remaining as they were)
      prefix = ((unsigned)window + found) << kWindowShift;
    } else {
      prefix = found;
    }
    remaining = sh.remaining;
    bits_left = shift;
    if (bits_left > 0 && sh.bucket <= kDirectMax) {  // few keys left: collect them, each finds its rank by counting
#pragma unroll
      for (int u = 0; u < kPer; ++u)
        if (u < mine && (in_window ? window_digit(x[u]) == found : (x[u] >> bits_left) == (prefix >> bits_left))) sh.list[atomicAdd(&sh.list_n, 1)] = x[u];
      __syncthreads();
      rank_finish(sh.list, sh.list_n, remaining, tid, &sh.threshold, &sh.need_eq);
      __syncthreads();
      prefix = sh.threshold;
      remaining = sh.need_eq;
      bits_left = 0;
    }
  }
  const unsigned T = prefix;
  const int need_eq = remaining;  // how many keys equal to T are kept: the lowest-index ones
  unsigned both = 0;              // keys above the threshold in the low half, keys equal to it in the high half
#pragma unroll
  for (int u = 0; u < kPer; ++u) both += u < mine ? (x[u] > T ? 1u : 0u) + (x[u] == T ? 0x10000u : 0u) : 0u;
  const unsigned before = sum_before<kWarps>(both, sh.warp_a, lane, warp);
  int gt = (int)(before & 0xFFFFu), eq = (int)(before >> 16);
  if (c == 0 && tid == kThreads - 1 && T == kProtectedKey && eq + (int)(both >> 16) > need_eq && device_status)
    atomicOr(device_status, FASTAV_DEV_PROTECT_OVERFLOW);  // more protected tokens than k
  if (kPer * tid == t0) sh.first_out = gt + min(eq, need_eq);   // t0 is a multiple of 16
  if (kPer * tid == t0 + m) sh.end_out = gt + min(eq, need_eq); // so is the end of a slice, but for the last one's
  if (kPer * tid >= t0 && kPer * tid < t0 + m) {
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const bool is_gt = x[u] > T, is_eq = x[u] == T;
      const int j = kPer * tid + u;
      if (u < mine && (is_gt || (is_eq && eq < need_eq))) {
        const int out = gt + min(eq, need_eq);
        if (out < room) keep_idx[base + out] = (global_idx ? tok0 : 0) + j;
        if (ROWS == kPlaces) a.place[tok0 + j] = out < room ? base + out : -1;
        picked[out & (kBins - 1)] = (unsigned)j;
      } else if (u < mine && ROWS == kPlaces) {
        a.place[tok0 + j] = -1;
      }
      gt += is_gt;
      eq += is_eq;
    }
  }
  if (a.do_gather && m > 0) {
    __syncthreads();
    first = sh.first_out;
    count = (t0 + m == n ? k : sh.end_out) - first;
  }
  }
  if (!a.do_gather || m == 0) return;  // (a block without tokens has nothing to copy)

  // ---- gather: this block's survivors, 16-byte chunks of all their rows dealt over the threads ---------------------
  __syncthreads();
  count = min(count, room - first);
  if constexpr (ROWS == kAhead) {
    if (a.rows.pos_in)
      for (int i = tid; i < count; i += kThreads) a.rows.pos_out[base + first + i] = pos_sh[picked[(first + i) & (kBins - 1)] - t0];
    if (rows_read())
      for (int i = warp - (kWarps - kRowWarps); i < count; i += kRowWarps)
        if (copies)
          bulk_store(piece.out + (long long)(base + first + i) * piece.out_stride,
                     ring + (picked[(first + i) & (kBins - 1)] - t0) * a.plan.row_bytes + piece.slot_off, piece.bytes);
    bulk_commit();
    bulk_wait_all();
    return;
  }
  const RowShape shape(s, a.rows);
  if (a.rows.pos_in)
    for (int i = tid; i < count; i += kThreads)
      a.rows.pos_out[base + first + i] = chain_load(a.rows.pos_in + tok0 + picked[(first + i) & (kBins - 1)]);
  const unsigned magic = 0xFFFFFFFFu / (unsigned)shape.n_chunks + 1u;  // e / n_chunks = umulhi(e, magic) while e * n_chunks < 2^32
  const int chunks = count * shape.n_chunks;
  const bool by_magic = shape.n_chunks > 1 && (long long)chunks * shape.n_chunks < 1ll << 32;  // (always, if max_keep holds: see little)
  constexpr int kUnroll = 6;
#pragma unroll 1
  for (int e0 = tid; e0 < chunks; e0 += kThreads * kUnroll) {
    uint4 v[kUnroll];
    int row[kUnroll], chunk[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int e = e0 + u * kThreads;
      if (e < chunks) {
        row[u] = by_magic ? (int)__umulhi((unsigned)e, magic) : e / shape.n_chunks;
        chunk[u] = e - row[u] * shape.n_chunks;
        v[u] = load_stream(chunk_in(s, a.rows, shape, (long long)tok0 + picked[(first + row[u]) & (kBins - 1)], chunk[u]));
      }
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      if (e0 + u * kThreads < chunks) store_row(chunk_out(s, a.rows, shape, (long long)base + first + row[u], chunk[u]), v[u]);
  }
}


int slice_of(const Shapes& s, int blocks) { return segment_of(s.max_seqlen) * (kSegments / blocks); }  // tokens per block

size_t smem_keys(const Shapes& s, int blocks) {
  return sizeof(FewShared) + few_layout(slice_of(s, blocks), s.hq * s.max_qlen, s.dim).total;
}

constexpr size_t kMaxDynamic = 220 * 1024;

// Tokens per block, at least (see cluster_blocks).  From the keys every token more per block counts: 32 tokens, sixteen blocks
// against eight, 1 x 512 tokens: 12.0 / 12.6 us, 1 x 2,048: 17.9 / 20.8; slices of 128 instead: 1 x 256 tokens 18.2 us instead of
// 12.2.  From sums or scores there is less to share and the exchange counts: with slices of 256 / 64 / 2,048 tokens the prune of 1 x
// 2,048 tokens, 32 rows, takes 20.7 / 22.9 / 23.9 us, 4 x 2,048 36.3 / 37.7 / 39.2.
constexpr int kKeySlice = 32, kScoreSlice = 256;
int cluster_keys(const Shapes& s) {
  int blocks = cluster_blocks(s.batch, s.max_seqlen, kKeySlice, s.cluster_limit);
  while (blocks < s.cluster_limit && smem_keys(s, blocks) > kMaxDynamic) blocks *= 2;
  return blocks;
}
int cluster_select(const Shapes& s) { return cluster_blocks(s.batch, s.max_seqlen, kScoreSlice, s.cluster_limit); }

template <Front FRONT, int DIM, Rows ROWS>
cudaError_t launch_kernel(const Shapes& s, const FewArgs& a, int blocks, size_t smem, const SelectArgs& t, cudaStream_t stream) {
  const auto kernel = prune_few_kernel<FRONT, DIM, ROWS>;
  cudaError_t e = once_per_context([&] {
    cudaError_t f = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxDynamic);
    if (f == cudaSuccess) f = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return f;
  });
  if (e != cudaSuccess) return e;
  e = launch_chained_cluster(kernel, dim3(s.batch * blocks), dim3(kThreads), blocks, smem, stream, s, a, t.cu_seqlens, t.keep_counts,
                             t.protect, t.q_idx, t.cu_qlens, t.keep_idx, t.cu_keep, t.device_status);
  count_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <Front FRONT, int DIM>
cudaError_t launch(const Shapes& s, FewArgs a, int blocks, size_t smem, const RowStreams* rows, const SelectArgs& t, cudaStream_t stream) {
  a.slice_cap = slice_of(s, blocks);
  a.place = t.place;
  // Four sequences and more, and a gather of few rows behind: that is as short as the launch of the next call's first kernel, which it is to hide
  // and which waits for this trigger first.  From the start / behind the keys, us: 16 x 60 rows of 12 KB, 60 % kept 15.3 / 18.1, 16 x 120 of 6 KB 16.2 / 18.6, 8
  // x 230 of 12 KB, 30 % 15.6 / 17.7.  Up to three sequences start late by 0.1 sooner.
  a.early = FRONT == kKeys && (!a.do_select || (!rows && !a.place && s.batch >= 4));
  if (rows) {
    a.do_gather = 1;
    a.rows = *rows;
    a.plan = bulk_plan(s, *rows);
    const size_t at = align_up(smem, 128), all = at + (size_t)a.slice_cap * (a.plan.row_bytes + sizeof(int));
    if (FRONT == kKeys && 2ll * s.total_keep >= s.total_tokens && a.plan.n_segments <= 32 && a.slice_cap <= kThreads && all <= kMaxDynamic) {
      a.ring = (int)at;
      smem = all;
    }
  }
  if constexpr (FRONT == kKeys) {
    if (a.place) return launch_kernel<FRONT, DIM, kPlaces>(s, a, blocks, smem, t, stream);
    if (a.ring) return launch_kernel<FRONT, DIM, kAhead>(s, a, blocks, smem, t, stream);
  }
  return launch_kernel<FRONT, DIM, kByList>(s, a, blocks, smem, t, stream);
}

template <Front FRONT>
cudaError_t launch_from(const Shapes& s, const FewArgs& a, const RowStreams* rows, const SelectArgs& t, cudaStream_t stream) {
  const int blocks = cluster_select(s);
  return launch<FRONT, 128>(s, a, blocks, sizeof(FewShared), rows, t, stream);
}

// Survivors' rows are copied by the blocks that select them where that is little per block: it saves a launch (tiny prompt of
// 512 tokens 10.3 us instead of 11.6), but the rows of one sequence then come through its own blocks only, and the compaction
// kernel has the whole chip (chain of 13 stages from 744 tokens: 162 us with limits of 0 and 48 KB, 241 with 192 KB).
// Survivors may all lie in one block's slice (early tokens are the ones attended to), so that has a limit too, a higher one
// where many sequences keep the chip busy.  Survivors spread / in one slice / rows by the compaction, from the keys: 1 x 1,024
// tokens of 1,536 bytes, 30 % kept (98 KB in one slice) 10.6 / 12.0 / 12.0 us, 1 x 2,048, 10 % (196 KB) 11.0 / 15.7 / 12.2, 16 x
// 2,000, 5 % (154 KB) 16.3 / 19.6 / 18.6.  From partial sums the blocks are fewer and one sequence does not gain: 1 x 512 tokens of
// 384 bytes, half kept 15.1 / 16.9 / 13.7; 8 x 1,000, 20 % 15.1 / 17.1 / 17.0, 16 x 2,000, 5 % 19.3 / 19.9 / 22.2, 256 x 128 of 640
// bytes, half kept 54 instead of 84.
constexpr int kGatherBytes = 48 << 10, kGatherBytesOneSlice = 96 << 10, kGatherBytesOneSliceBusy = 160 << 10;
bool little(const Shapes& s, int blocks, int row_bytes) {
  const int slice = slice_of(s, blocks);
  const long long spread = (s.max_keep + blocks - 1) / blocks, one_slice = s.max_keep < slice ? s.max_keep : slice;
  return row_bytes > 0 && spread * row_bytes <= kGatherBytes && one_slice * row_bytes <= (s.batch >= 16 ? kGatherBytesOneSliceBusy : kGatherBytesOneSlice);
}

}  // namespace

// Asked of the few-rows kernel with all the shared memory it may take (the one-pass score needs an SM per block too), once per
// context: a device with fewer SMs per GPC, or a context that was given a part of one, may have no room for sixteen.
int cluster_limit() {
  static std::atomic<unsigned long long> known[8];  // context number x 2 + (sixteen can be placed)
  static std::atomic<unsigned> next{0};
  const unsigned long long context = current_context();
  for (const auto& k : known) {
    const unsigned long long v = k.load(std::memory_order_acquire);
    if (context && v >> 1 == context) return v & 1 ? kMaxCluster : kPortableCluster;
  }
  const auto kernel = prune_few_kernel<kKeys, 128, kByList>;
  int clusters = 0;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxDynamic);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kMaxCluster);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kMaxDynamic;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = kMaxCluster;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    e = cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg);
  }
  if (e != cudaSuccess) (void)cudaGetLastError();
  const bool sixteen = e == cudaSuccess && clusters > 0;
  if (context && e == cudaSuccess)
    known[next.fetch_add(1, std::memory_order_relaxed) % 8].store(context << 1 | (sixteen ? 1u : 0u), std::memory_order_release);
  return sixteen ? kMaxCluster : kPortableCluster;
}

// Few scored rows, up to 2,048 tokens (kPer keys per thread).  More sequences than SMs take several rounds, one sequence per block:
// that is still the better way up to 512 tokens (300 x 128: 145 us, 600 x 200: 407; with the scoring kernels of long sequences
// 162 and 449), and no longer at 1,024 (160 x 1,024: 490 against 468, 300 x 1,024: 887 against 867).
bool few_applies(const Shapes& s) {
  if ((s.flags & FASTAV_SCORE_PATH_MASK) != 0) return false;
  if (s.max_qlen < 1 || s.max_qlen > kNarrowMaxRows || s.max_qlen * s.group > 128) return false;
  if (s.batch > kNumSMs && s.max_seqlen > 512) return false;
  return s.max_seqlen >= 1 && s.max_seqlen <= kMaxTokens && smem_keys(s, cluster_keys(s)) <= kMaxDynamic;
}
int few_blocks(const Shapes& s) { return s.batch * cluster_keys(s); }
bool cluster_select_applies(const Shapes& s) { return s.max_seqlen <= kMaxTokens; }

bool few_gathers(const Shapes& s, int row_bytes) { return little(s, cluster_keys(s), row_bytes); }
bool cluster_select_gathers(const Shapes& s, int row_bytes) { return s.batch >= 8 && little(s, cluster_select(s), row_bytes); }

cudaError_t launch_few(const Shapes& s, const void* q, const void* k, const float* lse_in, float* scores_out, bool do_select,
                       const RowStreams* rows, const SelectArgs& t, cudaStream_t stream) {
  FewArgs a{};
  a.q = static_cast<const uint16_t*>(q);
  a.k = static_cast<const uint16_t*>(k);
  a.lse = lse_in;
  a.scores_out = scores_out;
  a.rq = s.max_qlen;
  a.do_select = do_select ? 1 : 0;
  const int blocks = cluster_keys(s);
  return s.dim == 128 ? launch<kKeys, 128>(s, a, blocks, smem_keys(s, blocks), rows, t, stream)
                      : launch<kKeys, 64>(s, a, blocks, smem_keys(s, blocks), rows, t, stream);
}

cudaError_t launch_select_partials(const Shapes& s, const float* partial, const ScoreLeft& left, float* scores_out, const RowStreams* rows,
                                   const SelectArgs& t, cudaStream_t stream) {
  FewArgs a{};
  a.in = partial;
  a.row_chunks = left.row_chunks;
  a.rows_per_chunk = left.rows_per_chunk;
  a.scores_out = scores_out;
  a.do_select = 1;
  return launch_from<kPartials>(s, a, rows, t, stream);
}

cudaError_t launch_select_scores(const Shapes& s, const float* scores, const SelectArgs& t, cudaStream_t stream) {
  FewArgs a{};
  a.in = scores;
  a.do_select = 1;
  return launch_from<kScores>(s, a, nullptr, t, stream);
}

}  // namespace fastav
