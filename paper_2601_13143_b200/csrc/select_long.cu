// What follows the scoring kernels on sequences of more than 2,048 tokens, in one kernel: the tensor-core sweeps' sums per (KV head,
// chunk of query rows) and token, or few rows' logits and statistics, become scores, in their fixed order, and the k highest
// are selected (Section 2.2; ties to the lower index, protected tokens always).  One thread-block cluster per sequence, a slice of
// at most 2,048 tokens per block.
//
// The keys stay where they are.  A pass takes 11 bits: each block counts its slice's digits, adds the bins it has to the block that
// owns them (distributed shared memory), and after a cluster barrier each reads all totals and finds the bin of the k-th largest
// for itself.  Where that bin holds at most 192 keys the blocks send one another theirs and how many they have above the bin, and each
// ranks them all by counting, else the next pass follows.  From that each block also knows what the blocks before it keep.
//
// Bound: latency, a chain of a dozen steps of which three are cluster barriers; from the wait to the end 8.3 us (3 x 8,001-9,001 tokens) to 9.2
// (4 x 16,384), of that 1 to 2.5 for the sums, 1.3 for the bins' exchange, 1.1 for the lists'.  13 bits from the first one on put 16
// bins on an octave instead of 32 (lists of 300 keys, 3.1 us to rank) and had four barriers: 12.5 us and 13; 13 bits of the window
// spread over more bins than their exchange pays for (2.2 to 3.3 us).  In calls, us: 3 x 8,001-9,001 tokens, log-sum-exp given 72.6 -> 69.2, 4 x 6,554 96.5 -> 95.1.
// It saves the kernel that added the sums up, and from logits those for statistics and scores.  Clusters of 4, 8 or 16 make no
// difference.  From finished scores (fastav_select) nothing is saved, and one block was quicker: 4 x 6,554 tokens 109.8 us against 111.7, 32
// ragged sequences 217.8 against 219.7 (calls that had finished scores then).
#include "cluster.cuh"
#include "common.cuh"
#include "row_stats.cuh"
#include "select_keys.cuh"

namespace fastav {
namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kPer = 4;                      // keys per thread
constexpr int kSlice = kPer * kThreads;      // most tokens of a block
constexpr int kDigitBits = 11;
constexpr int kBins = 1 << kDigitBits;
constexpr int kBinsPerThread = kBins / kThreads;  // two words of two counts
// Keys of a bin that are ranked by counting.  Their comparisons grow with the square, another pass over the bits costs 2 us whatever its keys:
// 1 x 3,633 tokens, 23 rows, some 240 / 300 / 400 keys in the bin with a limit of 512 22.1 / 24.9 / 28.1 us, with 192 21.8 (with 128 some more
// calls pay the pass: 21.8 instead of 21.3 at 150 keys).
constexpr int kListMax = 192;
constexpr int kMaxTerms = 256 * kNarrowMaxRows;  // heads x scored rows of the few-rows path
// Shared memory that a block asks for, so that no block of a compaction with full rings (192 KB; fewer survivors make shorter ones) is resident
// beside it: those wait for the selection and slow it down.  Together with the successor started ahead of the passes instead of first thing: 32 ragged
// sequences of up to 8,192 tokens 307 -> 301 us, 4 x 16,384 292 -> 288.
constexpr size_t kLeastBytes = 64 * 1024;
constexpr int kSent = 32;                    // keys that a block sends to the others
constexpr int kLeastSlice = 256;             // tokens per block worth a block

// Two counts to a word: a slice has at most 2,048 keys, a sequence at most 32,768.
struct alignas(16) LongShared {
  union {
    unsigned hist[kBins / 2];          // of the block's slice
    unsigned sent[kMaxCluster][kSent]; // what the cluster's blocks have in their lists
    unsigned all[kListMax];            // ... fetched from where it lies
  };
  unsigned prot_bits[kSlice / 32];
  unsigned list[kListMax];
  unsigned warp_a[kWarps], warp_b[kWarps];
  unsigned count_of[kMaxCluster];  // keys in each block's list (low half), keys above the list's bin (high half)
  unsigned kept_of[kMaxCluster];   // keys above the threshold (low half) and on it (high half)
  int index[8];
  int base, list_n, remaining, bucket, need_eq;
  unsigned prefix, threshold, own, above_n, earlier;
};

enum Front { kPartials, kLogits };

struct LongArgs {
  const float* in;                 // kPartials [Hkv * row_chunks][N]; kLogits [Hq * rq][N]
  int row_chunks, rows_per_chunk;  // kPartials
  const float2* stats;             // kLogits [total_q * Hq][stat_tiles]
  const float* lse_in;             // kLogits, optional: the caller's natural-log log-sum-exp [total_q, Hq], in place of stats
  int rq, stat_tiles;              // kLogits: most scored rows of a sequence
  float* scores_out;
  int blocks, slice_cap;           // blocks of a cluster; tokens of a block that the longest sequence needs
};

// After LongShared: the scores of the slice, then the totals of the bins this block owns, of the whole cluster.
__host__ __device__ inline int owned_words(int blocks) { return kBins / 2 / blocks; }
static_assert(kBins / 2 / kMaxCluster % 4 == 0, "cleared 16 bytes at a time");
// ... and of kLogits what each term's weights are made with, at most `terms`.
inline size_t long_bytes(int blocks, int slice_cap, int terms) {
  const size_t used = sizeof(LongShared) + (size_t)(slice_cap + owned_words(blocks) + 2 * terms) * sizeof(unsigned);
  return used > kLeastBytes ? used : kLeastBytes;
}
template <int N>
struct Tokens {
  static constexpr int value = N;
};
__host__ __device__ inline int slice_for(int n, int blocks) { return ((n + blocks - 1) / blocks + 31) & ~31; }

__device__ __forceinline__ void remote_add(uint32_t a, unsigned v) {
  asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned remote_load(uint32_t a) {
  unsigned v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint2 remote_load2(uint32_t a) {  // 8-byte aligned
  uint2 v;
  asm volatile("ld.shared::cluster.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
  return v;
}

// rank_finish for a list that may be longer: lanes of a warp share a key where the block has more threads than there are keys, each
// compares it with every so many quads (300 keys: 3.1 us one after the other).
__device__ __forceinline__ void rank_list(const unsigned* list, int count, int remaining, int tid, unsigned* threshold, int* need_eq) {
  const int log_lanes = min(5, 31 - __clz(kThreads) - (32 - __clz(count - 1))), lanes = 1 << log_lanes;  // lanes x count <= kThreads
  const int at = tid >> log_lanes, part = tid & (lanes - 1), whole = count >> 2;
  const bool active = at < count;
  const unsigned mine = active ? list[at] : 0u;
  int both = 0;  // keys above in the high half, equal ones in the low half
  if (active) {
#pragma unroll 2
    for (int i = part; i < whole; i += lanes) {
      const uint4 v = *reinterpret_cast<const uint4*>(list + 4 * i);
      both += (v.x > mine ? 0x10000 : 0) + (v.y > mine ? 0x10000 : 0) + (v.z > mine ? 0x10000 : 0) + (v.w > mine ? 0x10000 : 0);
      both += (v.x == mine) + (v.y == mine) + (v.z == mine) + (v.w == mine);
    }
    for (int i = 4 * whole + part; i < count; i += lanes) both += (list[i] > mine ? 0x10000 : 0) + (list[i] == mine);
  }
  __syncwarp();
  for (int d = lanes / 2; d; d >>= 1) both += __shfl_xor_sync(0xFFFFFFFFu, both, d);
  const int above = both >> 16, equal = both & 0xFFFF;
  if (active && part == 0 && above < remaining && remaining <= above + equal) {
    *threshold = mine;
    *need_eq = remaining - above;
  }
}

template <Front FRONT>
__global__ void __launch_bounds__(kThreads, 1) select_long_kernel(Shapes s, LongArgs a, const int32_t* __restrict__ cu_seqlens,
                                                                  const int32_t* __restrict__ keep_counts, const uint8_t* __restrict__ protect,
                                                                  const int32_t* __restrict__ q_idx, const int32_t* __restrict__ cu_qlens,
                                                                  int32_t* __restrict__ keep_idx, int32_t* __restrict__ cu_keep, int32_t* device_status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  LongShared& sh = *reinterpret_cast<LongShared*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int blocks = a.blocks, b = (int)blockIdx.x / blocks, c = (int)cluster_rank();
  unsigned* const keys = reinterpret_cast<unsigned*>(smem_raw + sizeof(LongShared));
  unsigned* const totals = keys + a.slice_cap;
  const int owned = owned_words(blocks);  // of an owner: a power of two, at least 64 words
  auto clear_counts = [&] {
    for (int i = tid; i < kBins / 8; i += kThreads) reinterpret_cast<uint4*>(sh.hist)[i] = make_uint4(0, 0, 0, 0);
    for (int i = tid; i < owned / 4; i += kThreads) reinterpret_cast<uint4*>(totals)[i] = make_uint4(0, 0, 0, 0);
  };
  clear_counts();
  if (tid < kSlice / 32) sh.prot_bits[tid] = 0u;
  if (tid == 0) { sh.base = 0; sh.list_n = 0; sh.above_n = 0u; sh.earlier = 0u; }
  cluster_arrive();  // this block runs and its totals are zero: waited for before the first remote access
  chain_enter_late(s, cu_seqlens, keep_counts, protect, q_idx, cu_qlens);
  if (warp == 0) {
    const int32_t* word = lane < 2 ? cu_seqlens + b + lane : lane < 4 ? cu_qlens + b + lane - 2 : keep_counts + b;
    if (lane < 5) sh.index[lane] = chain_load(word);
  }
  __syncthreads();
  const Span seq = checked_words(sh.index[0], sh.index[1], s.total_tokens, s.max_seqlen);
  const Span qrows = checked_words(sh.index[2], sh.index[3], s.total_q, s.max_qlen);
  int k = sh.index[4];
  const bool k_clamped = k < 0 || k > seq.count;
  const int tok0 = seq.first, n = min(seq.count, a.slice_cap * blocks);
  const int slice = slice_for(n, blocks), t0 = min(n, c * slice), m = min(n - t0, slice);
  k = k < 0 ? 0 : (k > n ? n : k);
  const bool lowest = (s.flags & FASTAV_SELECT_LOWEST) != 0;

  {  // ahead of the wait: the output offset, the clamped keep counts of the sequences before this one, 32 per warp
    if (warp * 32 < b) {
      int part = 0;
#pragma unroll 1
      for (int i = warp * 32 + lane; i < b; i += kThreads) {
        const int ni = seq_span(s, cu_seqlens, i).count, ki = chain_load(keep_counts + i);
        part += ki < 0 ? 0 : min(ki, ni);
      }
      part = __reduce_add_sync(0xFFFFFFFFu, part);
      if (lane == 0 && part) atomicAdd(&sh.base, part);
    }
    if (s.flags & FASTAV_PROTECT_QUERY_ROWS)
      for (int r = tid; r < qrows.count; r += kThreads) {
        const int j = chain_load(q_idx + qrows.first + r) - t0;  // relative to this block's first token
        if (j >= 0 && j < m) atomicOr(&sh.prot_bits[j >> 5], 1u << (j & 31));
      }
    if (protect)
      for (int j0 = warp * 32; j0 < m; j0 += kThreads) {  // a warp covers 32 tokens: one word
        const int j = j0 + lane;
        const unsigned word = __ballot_sync(0xFFFFFFFFu, j < m && chain_load(protect + tok0 + t0 + j) != 0);
        if (lane == 0 && word) atomicOr(&sh.prot_bits[j0 >> 5], word);
      }
  }
  pdl_wait();
  const float* in = a.in;
  pdl_acquire(in);
  if (tid == 0 && c == 0 && device_status) {
    if (seq.bad || qrows.bad) atomicOr(device_status, FASTAV_DEV_SHAPE_MISMATCH);
    if (k_clamped) atomicOr(device_status, FASTAV_DEV_K_CLAMPED);
  }
  const float* const col = in + tok0 + t0;
  const int rows = FRONT == kLogits ? min(qrows.count, a.rq) : 0, terms = s.hq * rows;  // term i = (head i / rows, row i % rows)
  float2* const weight = reinterpret_cast<float2*>(totals + owned);
  const float2* stats = a.stats;
  if constexpr (FRONT == kLogits) pdl_acquire(stats);
  auto merge_stats = [&] {
    if constexpr (FRONT == kLogits) {
      const int l16 = lane & (kMergeLanes - 1), tiles = (n + kRowTileTokens - 1) / kRowTileTokens;
#pragma unroll 1
      for (int i0 = 0; i0 < terms; i0 += kThreads / kMergeLanes) {
        const int i = i0 + tid / kMergeLanes, head = i / rows, r = i - head * rows;
        const long long at = (long long)(qrows.first + r) * s.hq + head;
        float2 w;
        if (a.lse_in) {
          const float v = i < terms ? chain_load(a.lse_in + at) : 0.f;
          w = weight_from_lse((v == v && fabsf(v) != INFINITY) ? v * kLog2e : INFINITY);  // a row that sees no key adds 0
        } else {
          w = weight_from_pair(merge_row_stats(stats + at * a.stat_tiles, i < terms ? tiles : 0, l16));
        }
        if (l16 == 0 && i < terms) weight[i] = w;
      }
      __syncthreads();
    }
  };
  // A thread's tokens lie kThreads apart; up to four of them are added up together.
  auto add_up = [&](auto tokens) {
    constexpr int kTokens = decltype(tokens)::value;
    auto have_from = [&](int j0) { return min(kTokens, (m - j0 + kThreads - 1) / kThreads); };
    Weights<kTokens> w;
    if constexpr (FRONT == kLogits) {  // the first logits are on their way while the statistics are merged
      w.fetch(col + tid, kThreads, have_from(tid), 0, terms, s.total_tokens);
      merge_stats();
    }
#pragma unroll 1
    for (int j0 = tid; j0 < m; j0 += kThreads * kTokens) {
      const int have = have_from(j0);
      float total[kTokens];
      if constexpr (FRONT == kPartials) {
        const int row_chunks = (qrows.count * s.group + a.rows_per_chunk - 1) / a.rows_per_chunk;
        sum_of_partials<32 / kTokens>(col + j0, kThreads, have, s.hkv, row_chunks, a.row_chunks, s.total_tokens, total);
        const float inv = qrows.count > 0 ? 1.0f / ((float)s.hq * (float)qrows.count) : 0.f;
#pragma unroll
        for (int t = 0; t < kTokens; ++t) total[t] *= inv;
      } else {
#pragma unroll
        for (int t = 0; t < kTokens; ++t) total[t] = 0.f;
#pragma unroll 1
        for (int i0 = 0; i0 < terms; i0 += w.kUnroll) {
          if (j0 != tid || i0 > 0) w.fetch(col + j0, kThreads, have, i0, terms, s.total_tokens);
          w.add(weight, i0, terms, total);
        }
#pragma unroll
        for (int t = 0; t < kTokens; ++t) total[t] = rows > 0 ? total[t] / ((float)s.hq * (float)qrows.count) : 0.f;
      }
#pragma unroll
      for (int t = 0; t < kTokens; ++t)
        if (t < have) {
          a.scores_out[tok0 + t0 + j0 + t * kThreads] = total[t];
          keys[j0 + t * kThreads] = __float_as_uint(total[t]);
        }
    }
  };
  if (m <= kThreads) add_up(Tokens<1>{});
  else if (m <= 2 * kThreads) add_up(Tokens<2>{});
  else add_up(Tokens<4>{});
  __syncthreads();
  const int base = sh.base;
  if (c == 0 && tid == 0) {
    cu_keep[b + 1] = base + k;
    if (b == 0) cu_keep[0] = 0;
    if (base + k > s.total_keep && device_status) atomicOr(device_status, FASTAV_DEV_SHAPE_MISMATCH);
  }
  // Thread t owns the tokens 4 t .. 4 t + 3 of the slice.
  const int mine = max(0, min(kPer, m - kPer * tid));
  unsigned x[kPer];
  {
    uint4 v = make_uint4(0, 0, 0, 0);
    if (mine > 0) v = *reinterpret_cast<const uint4*>(&keys[kPer * tid]);
    const unsigned raw[kPer] = {v.x, v.y, v.z, v.w}, prot = sh.prot_bits[tid / (32 / kPer)] >> (kPer * (tid % (32 / kPer)));
    bool any_protected = false;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const float score = __uint_as_float(raw[u]);
      x[u] = order_key(lowest ? -score : score);
      if (x[u] == kProtectedKey) x[u] = kProtectedKey - 1;  // only a NaN pattern lands here
      if ((prot >> u) & 1u) x[u] = kProtectedKey;
      any_protected |= u < mine && x[u] == kProtectedKey;
    }
    if (k == 0 && any_protected && device_status) atomicOr(device_status, FASTAV_DEV_PROTECT_OVERFLOW);
  }
  cluster_wait();
  if (k == 0) return;  // nothing is kept, protected or not (uniform for the cluster; nothing remote has been touched)

  pdl_trigger();
  // The first pass looks at scores from 2^-63 up to 2 only: three leading bits are the same there, so that a bin is 1/32 of an octave
  // wide instead of 1/4, and the bin of the k-th largest holds few keys.  Smaller scores share the lowest bin, larger ones
  // (and protected tokens) the highest; where the k-th largest lies in one of these two among many, the passes start again from the first bit.
  constexpr int kWindowShift = 29 - kDigitBits;  // three leading bits, then the digit
  const int window = lowest ? 2 << kDigitBits : 5 << kDigitBits;
  auto window_digit = [&](unsigned key) { return (unsigned)min(max((int)(key >> kWindowShift) - window, 0), kBins - 1); };
  bool windowed = true;
  unsigned prefix = 0u;  // the bits of the k-th largest key fixed so far
  int remaining = k, bits_left = 32;
  bool listed = false;   // the threshold comes from the cluster's list
  bool pulls = false;    // ... which was fetched
  unsigned list_key = 0u;
  int list_from = kMaxCluster;
#pragma unroll 1
  for (int pass = 0; bits_left > 0; ++pass) {
    const int shift = windowed ? kWindowShift : max(0, bits_left - kDigitBits);
    const unsigned above_want = __funnelshift_rc(prefix, 0u, bits_left);  // prefix >> bits_left, 0 for 32
    if (pass > 0) {
      cluster_sync();  // everybody has read the totals
      clear_counts();
      cluster_sync();
    }
    {
      unsigned run_digit = kBins, run_len = 0u;  // equal digits of consecutive tokens (typically zeros): one update
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        if (u < mine && __funnelshift_rc(x[u], 0u, bits_left) == above_want) {
          const unsigned digit = windowed ? window_digit(x[u]) : (x[u] >> shift) & (kBins - 1);
          if (digit != run_digit) {
            if (run_len) atomicAdd(&sh.hist[run_digit >> 1], run_len << (16 * (run_digit & 1)));
            run_digit = digit;
            run_len = 0u;
          }
          ++run_len;
        }
      }
      if (run_len) atomicAdd(&sh.hist[run_digit >> 1], run_len << (16 * (run_digit & 1)));
    }
    __syncthreads();
    constexpr int kWords = kBinsPerThread / 2;
    static_assert(kWords == 2);
    const int first_word = tid * kWords, owner = first_word / owned;
    const uint32_t owner_at = remote(&totals[first_word & (owned - 1)], owner);
    {
      const uint2 v = *reinterpret_cast<const uint2*>(&sh.hist[first_word]);
      if (v.x) remote_add(owner_at, v.x);
      if (v.y) remote_add(owner_at + 4, v.y);
    }
    cluster_sync();
    unsigned h[kBinsPerThread], own = 0;
    {
      const uint2 v = remote_load2(owner_at);
      h[0] = v.x & 0xFFFFu;
      h[1] = v.x >> 16;
      h[2] = v.y & 0xFFFFu;
      h[3] = v.y >> 16;
    }
#pragma unroll
    for (int i = 0; i < kBinsPerThread; ++i) own += h[i];
    unsigned above = sum_above<kWarps>(own, sh.warp_a, lane, warp);
    const unsigned rem = (unsigned)remaining;
    if (above < rem && rem <= above + own) {  // exactly one thread: its bins from the top
#pragma unroll
      for (int i = kBinsPerThread - 1; i >= 0; --i) {
        if (above < rem && rem <= above + h[i]) {
          sh.prefix = windowed ? (unsigned)(2 * first_word + i) : prefix | ((unsigned)(2 * first_word + i) << shift);
          sh.remaining = (int)(rem - above);
          sh.bucket = (int)h[i];
        }
        above += h[i];
      }
    }
    __syncthreads();
    const unsigned found = sh.prefix;
    const int bucket = sh.bucket;
    const bool in_window = windowed;
    if (windowed) {
      windowed = false;
      if ((found == 0u || found == kBins - 1) && bucket > kListMax) continue;  // (prefix and remaining as they were)
      prefix = ((unsigned)window + found) << kWindowShift;
    } else {
      prefix = found;
    }
    remaining = sh.remaining;
    bits_left = shift;
    if (bits_left > 0 && bucket <= kListMax) {  // few keys left in the cluster: everybody fetches them and finds their ranks by counting
      unsigned over = 0u;
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const unsigned digit = in_window ? window_digit(x[u]) : x[u] >> bits_left, wanted = in_window ? found : prefix >> bits_left;
        if (u < mine && digit == wanted) sh.list[atomicAdd(&sh.list_n, 1)] = x[u];
        over += u < mine && digit > wanted;
      }
      over = __reduce_add_sync(0xFFFFFFFFu, over);
      if (lane == 0 && over) atomicAdd(&sh.above_n, over);
      __syncthreads();
      const int here = sh.list_n;
      if (tid < blocks) remote_store(remote(&sh.count_of[c], tid), (unsigned)here | sh.above_n << 16);
      if (here <= kSent)
        for (int i = tid; i < here * blocks; i += kThreads) remote_store(remote(&sh.sent[c][i / blocks], i & (blocks - 1)), sh.list[i / blocks]);
      cluster_sync();
      const int count = lane < blocks ? (int)(sh.count_of[lane] & 0xFFFFu) : 0;
      const unsigned* ranked = sh.list;
      pulls = __any_sync(0xFFFFFFFFu, count > kSent);  // (the same for the whole cluster)
      if (!pulls) {  // warp w has block w's
        const int start = (int)__reduce_add_sync(0xFFFFFFFFu, lane < warp ? count : 0), own = __shfl_sync(0xFFFFFFFFu, count, warp & 31);
        if (lane < own) {
          list_key = sh.sent[warp][lane];
          list_from = warp;
          sh.list[start + lane] = list_key;
        }
      } else {
        if (tid < bucket) {
          int at = tid, from = 0;
          while (from < blocks - 1 && at >= (int)(sh.count_of[from] & 0xFFFFu)) at -= (int)(sh.count_of[from++] & 0xFFFFu);
          list_key = remote_load(remote(&sh.list[min(at, kListMax - 1)], from));
          list_from = from;
          sh.all[tid] = list_key;
        }
        cluster_arrive();  // nothing remote from here on: waited for before the block may exit
        ranked = sh.all;
      }
      __syncthreads();
      rank_list(ranked, bucket, remaining, tid, &sh.threshold, &sh.need_eq);
      __syncthreads();
      prefix = sh.threshold;
      remaining = sh.need_eq;
      bits_left = 0;
      listed = true;
    }
  }
  const unsigned T = prefix;
  const int need_eq = remaining;  // how many keys equal to T are kept: the lowest-index ones
  unsigned both = 0;              // keys above the threshold in the low half, keys equal to it in the high half
#pragma unroll
  for (int u = 0; u < kPer; ++u) both += u < mine ? (x[u] > T ? 1u : 0u) + (x[u] == T ? 0x10000u : 0u) : 0u;
  // The blocks before this one: how many of theirs lie above and on the threshold.  From the list and the counts beside it every
  // block works that out for itself; without a list they tell one another.
  if (listed) {
    unsigned part = list_from < c ? (list_key > T ? 1u : 0u) + (list_key == T ? 0x10000u : 0u) : 0u;
    if (warp == 0 && lane < c) part += sh.count_of[lane] >> 16;
    part = __reduce_add_sync(0xFFFFFFFFu, part);
    if (lane == 0 && part) atomicAdd(&sh.earlier, part);
  }
  const unsigned before = sum_before<kWarps>(both, sh.warp_b, lane, warp);
  unsigned earlier;
  if (listed) {
    earlier = sh.earlier;
  } else {
    if (tid == kThreads - 1) sh.own = before + both;
    __syncthreads();
    if (tid < blocks) remote_store(remote(&sh.kept_of[c], tid), sh.own);
    cluster_sync();  // the last remote access
    earlier = __reduce_add_sync(0xFFFFFFFFu, lane < c ? sh.kept_of[lane] : 0u);
  }
  int gt = (int)(before & 0xFFFFu) + (int)(earlier & 0xFFFFu);
  int eq = (int)(before >> 16) + (int)(earlier >> 16);
  if (T == kProtectedKey) {  // more protected tokens than k? (uniform for the block)
    const int all_eq = listed ? __syncthreads_count(list_from < kMaxCluster && list_key == T) : sh.bucket;
    if (c == 0 && tid == 0 && all_eq > need_eq && device_status) atomicOr(device_status, FASTAV_DEV_PROTECT_OVERFLOW);
  }
  const int offset = ((s.flags & FASTAV_KEEP_IDX_GLOBAL) ? tok0 : 0) + t0 + kPer * tid;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const bool is_gt = u < mine && x[u] > T, is_eq = u < mine && x[u] == T;
    const int out = base + gt + min(eq, need_eq);
    if ((is_gt || (is_eq && eq < need_eq)) && out < s.total_keep) keep_idx[out] = offset + u;
    gt += is_gt;
    eq += is_eq;
  }
  if (pulls) cluster_wait();
}

// Blocks per sequence, as many as run at once and have a slice worth it; 0 where the longest sequence does not fit.
int blocks_for(const Shapes& s) {
  const int blocks = cluster_blocks(s.batch, s.max_seqlen, kLeastSlice, s.cluster_limit);
  return blocks >= 2 && slice_for(s.max_seqlen, blocks) <= kSlice ? blocks : 0;
}

}  // namespace

bool long_select_applies(const Shapes& s) { return !cluster_select_applies(s) && blocks_for(s) > 0; }

namespace {

template <Front FRONT>
cudaError_t launch(const Shapes& s, LongArgs a, float* scores_out, const SelectArgs& t, cudaStream_t stream) {
  a.scores_out = scores_out;
  a.blocks = blocks_for(s);
  a.slice_cap = slice_for(s.max_seqlen, a.blocks);
  const int terms = FRONT == kLogits ? s.hq * a.rq : 0;
  cudaError_t e = once_per_context([] {
    const cudaError_t f = cudaFuncSetAttribute(select_long_kernel<FRONT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)long_bytes(2, kSlice, FRONT == kLogits ? kMaxTerms : 0));
    return f == cudaSuccess ? cudaFuncSetAttribute(select_long_kernel<FRONT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) : f;
  });
  if (e != cudaSuccess) return e;
  e = launch_chained_cluster(select_long_kernel<FRONT>, dim3(s.batch * a.blocks), dim3(kThreads), a.blocks, long_bytes(a.blocks, a.slice_cap, terms), stream,
                             s, a, t.cu_seqlens, t.keep_counts, t.protect, t.q_idx, t.cu_qlens, t.keep_idx, t.cu_keep, t.device_status);
  count_launches(1);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

cudaError_t launch_long_partials(const Shapes& s, const float* partial, const ScoreLeft& left, float* scores_out, const SelectArgs& t, cudaStream_t stream) {
  LongArgs a{};
  a.in = partial;
  a.row_chunks = left.row_chunks;
  a.rows_per_chunk = left.rows_per_chunk;
  return launch<kPartials>(s, a, scores_out, t, stream);
}

cudaError_t launch_long_logits(const Shapes& s, const Workspace& w, const unsigned char* ws, const float* lse_in, float* scores_out, const SelectArgs& t,
                               cudaStream_t stream) {
  LongArgs a{};
  a.in = reinterpret_cast<const float*>(ws + w.logits_off);
  a.stats = reinterpret_cast<const float2*>(ws + w.stats_off);
  a.lse_in = lse_in;
  a.rq = s.max_qlen;
  a.stat_tiles = w.stat_tiles;
  return launch<kLogits>(s, a, scores_out, t, stream);
}

}  // namespace fastav
