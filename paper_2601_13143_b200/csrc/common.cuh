// Internal declarations shared by the kernels and the C-ABI layer.  Nothing here is exported.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

#include "fastav.h"

namespace fastav {

constexpr int kNumSMs = 148;          // B200: 2 dies x 74 SMs; grids are sized in multiples of this
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// Device-side view of one call's shapes (a trimmed fastav_params, passed by value).
struct Shapes {
  int batch, total_tokens, max_seqlen, total_q, max_qlen, total_keep, max_keep;
  int hq, hkv, group, dim, hidden;
  long long q_st, q_sh, k_st, k_sh, v_st, v_sh, ko_st, ko_sh, vo_st, vo_sh;
  float scale_log2;  // softmax scale * log2(e): logits are kept in base-2 units
  unsigned flags;
  int cluster_limit; // most blocks of a cluster in the current context (host side)
  int head_wait;     // set at launch (launch_chained): this kernel opens a call and must wait before it reads anything
};

// For the kernels that take no Shapes: the same mark.
struct ChainHead { int head_wait = 0; };

// What a prune call still has to do after the scoring kernels, and from what.
struct ScoreLeft {
  enum Kind { kScores, kKeys, kPartials, kLogits } kind = kScores;  // finished scores; nothing done: the kernel that selects starts
                                                                     // from the keys; sums per (KV head, chunk of query rows) and
                                                                     // token; logits and statistics of few rows
  int row_chunks = 0, rows_per_chunk = 0;                   // kPartials: most chunks of a KV head, query rows of a chunk
};

// Carved from the caller's workspace by plan_workspace(); all offsets 256-byte aligned.
struct Workspace {
  size_t total = 0;
  // generic / narrow score
  size_t stats_off = 0;     // float2 [total_q * Hq][stat_tiles]   per-tile (max, sum-exp2)
  size_t lse_off = 0;       // float  [total_q * Hq]               log2-sum-exp2 per (row, head)
  size_t partial_off = 0;   // float  [Hkv * row chunks][N]        score partials per KV head and chunk of query rows
  size_t logits_off = 0;    // float  [Hq][max_qlen][N] (matrix-vector path only; 0 bytes otherwise)
  // select
  size_t keys_off = 0;      // uint32 [N] (only when a sequence does not fit in shared memory); a prune call: a token's place among the survivors
  int stat_tiles = 0;
};

Workspace plan_workspace(const fastav_params& p);
Shapes make_shapes(const fastav_params& p);

// ---- launchers (each returns cudaGetLastError() after its launches) -------------------------
cudaError_t launch_score(const Shapes& s, const Workspace& w, const void* q, const int32_t* q_idx,
                         const int32_t* cu_qlens, const void* k, const int32_t* cu_seqlens, const float* lse_in,
                         float* scores_out, unsigned char* ws, int32_t* device_status, cudaStream_t stream, ScoreLeft* left = nullptr);

// `left` (optional, everywhere below): when given, a launcher may leave work to the kernel that selects and say what;
// without it the scores are finished.
// `lse_in` (optional, everywhere below): the caller's natural-log log-sum-exp per (scored row, head); when
// given, the softmax statistics are not recomputed.
cudaError_t launch_score_generic(const Shapes& s, const Workspace& w, const void* q, const int32_t* q_idx,
                                 const int32_t* cu_qlens, const void* k, const int32_t* cu_seqlens, const float* lse_in,
                                 float* scores_out, unsigned char* ws, cudaStream_t stream);

// lse_ws[i] = log2(e) * lse_in[i] (the kernels work in base-2 units); a non-finite entry (a row that saw no
// key) becomes +inf, i.e. the row contributes nothing.
cudaError_t launch_lse_import(const Shapes& s, const float* lse_in, float* lse_ws, cudaStream_t stream);
// ... and back: the workspace's statistics as natural-log log-sum-exp [total_q, Hq] (-inf where a row sees no key).
cudaError_t launch_lse_export(const Shapes& s, const float* lse_ws, float* lse_out, cudaStream_t stream);

// Few scored rows per sequence (the paper's fine stage scores the last token only): matrix-vector path.
constexpr int kNarrowMaxRows = 4;
bool score_narrow_applies(const Shapes& s);
cudaError_t launch_score_narrow(const Shapes& s, const Workspace& w, const void* q, const int32_t* q_idx,
                                const int32_t* cu_qlens, const void* k, const int32_t* cu_seqlens, const float* lse_in,
                                float* scores_out, unsigned char* ws, int32_t* device_status, cudaStream_t stream, ScoreLeft* left);

// Many scored rows per sequence: tensor-core path (tcgen05 + TMA).  `*used` is false when the TMA
// descriptor for K could not be built; nothing was launched then and the caller takes another path.
int wide_rows_per_chunk(int group);
int wide_row_chunks(int max_qlen, int group);
bool score_wide_applies(const Shapes& s);
cudaError_t launch_score_wide(const Shapes& s, const Workspace& w, const void* q, const int32_t* q_idx,
                              const int32_t* cu_qlens, const void* k, const int32_t* cu_seqlens, const float* lse_in,
                              float* scores_out, unsigned char* ws, int32_t* device_status, cudaStream_t stream, bool* used, ScoreLeft* left);

// Few scored rows on longer sequences: logits and their statistics per 64 tokens (score_rows.cu); log-sum-exp per (row, head).
// `*used` is false when it does not take the shapes; nothing was launched then.
cudaError_t launch_rows(const Shapes& s, const Workspace& w, const void* q, const int32_t* q_idx, const int32_t* cu_qlens, const void* k,
                        const int32_t* cu_seqlens, unsigned char* ws, int32_t* device_status, cudaStream_t stream, bool* used);
cudaError_t launch_rows_lse(const Shapes& s, const Workspace& w, const int32_t* cu_qlens, const int32_t* cu_seqlens, unsigned char* ws,
                            cudaStream_t stream);

// The kernel that selects, a thread-block cluster per sequence (prune_few.cu): from the keys themselves (few scored rows, short
// sequences), from partial sums or from finished scores, to the keep list, or to the gathered rows.
struct RowStreams;
struct SelectArgs {
  const int32_t *cu_seqlens, *keep_counts;
  const uint8_t* protect;
  const int32_t *q_idx, *cu_qlens;
  int32_t *keep_idx, *cu_keep, *device_status;
  int32_t* place = nullptr;  // launch_few, optional, [N]: where a token's row goes among the survivors, -1 if it is dropped
};
int few_blocks(const Shapes& s);                // ... blocks of that kernel, each on an SM of its own as long as there are as many
bool few_applies(const Shapes& s);              // from the keys
bool cluster_select_applies(const Shapes& s);   // from partial sums or scores
bool few_gathers(const Shapes& s, int row_bytes);
bool cluster_select_gathers(const Shapes& s, int row_bytes);
// `rows`: what to gather in the same kernel (nullptr: nothing).
cudaError_t launch_few(const Shapes& s, const void* q, const void* k, const float* lse_in, float* scores_out, bool do_select,
                       const RowStreams* rows, const SelectArgs& t, cudaStream_t stream);
cudaError_t launch_select_partials(const Shapes& s, const float* partial, const ScoreLeft& left, float* scores_out, const RowStreams* rows,
                                   const SelectArgs& t, cudaStream_t stream);
cudaError_t launch_select_scores(const Shapes& s, const float* scores, const SelectArgs& t, cudaStream_t stream);

// ... and of longer sequences, a slice of the tokens per block (select_long.cu), from partial sums or from logits.
bool long_select_applies(const Shapes& s);
cudaError_t launch_long_partials(const Shapes& s, const float* partial, const ScoreLeft& left, float* scores_out, const SelectArgs& t, cudaStream_t stream);
cudaError_t launch_long_logits(const Shapes& s, const Workspace& w, const unsigned char* ws, const float* lse_in, float* scores_out, const SelectArgs& t,
                               cudaStream_t stream);

// Most blocks of a cluster that the current context can place: 16, or the portable 8.
int cluster_limit();

// Many scored rows on short sequences: one pass over K (score_once.cu).
struct OncePlan {
  int rows_per_tile, row_tiles, blocks, tiles_per_block, rounds;
};
constexpr int kOnceMaxTokens = 4096;
int once_row_tiles(int max_qlen, int group);
bool once_plan(const Shapes& s, bool lse_given, OncePlan* plan);
cudaError_t launch_score_once(const Shapes& s, const void* k_map, const void* q_map, const int32_t* q_idx, const int32_t* cu_qlens,
                              const int32_t* cu_seqlens, const float* lse_in, const OncePlan& plan, float* partial, int32_t* device_status,
                              cudaStream_t stream);

cudaError_t launch_select(const Shapes& s, const Workspace& w, const float* scores, const int32_t* cu_seqlens,
                          const int32_t* keep_counts, const uint8_t* protect, const int32_t* q_idx,
                          const int32_t* cu_qlens, int32_t* keep_idx, int32_t* cu_keep, unsigned char* ws,
                          int32_t* device_status, cudaStream_t stream);

cudaError_t launch_compact(const Shapes& s, const int32_t* keep_idx, const int32_t* cu_keep,
                           const int32_t* cu_seqlens, const void* hidden_in, void* hidden_out, const int32_t* pos_in,
                           int32_t* pos_out, const void* k_in, void* k_out, const void* v_in, void* v_out,
                           int32_t* device_status, cudaStream_t stream);

// The same for a call whose rows shared memory holds, behind launch_few: they are read while that kernel selects, which leaves every
// token's place for it (SelectArgs::place).
bool placed_compact_applies(const Shapes& s, const RowStreams& rows);
cudaError_t launch_compact_placed(const Shapes& s, const RowStreams& rows, const int32_t* place, const int32_t* cu_seqlens, int32_t* device_status,
                                  cudaStream_t stream);

int32_t validate_prune(const fastav_params* params, const void* q, const int32_t* q_idx, const int32_t* cu_qlens, const void* k,
                       const void* v, const int32_t* cu_seqlens, const int32_t* keep_counts, const void* hidden_in,
                       const int32_t* pos_in, const float* scores_out, const int32_t* keep_idx_out, const int32_t* cu_keep_out,
                       const void* hidden_out, const int32_t* pos_out, const void* k_out, const void* v_out, const void* workspace,
                       size_t workspace_bytes);

cudaError_t enqueue_selection(const fastav_params& params, const void* q, const int32_t* q_idx, const int32_t* cu_qlens, const void* k,
                              const int32_t* cu_seqlens, const float* lse_opt, const int32_t* keep_counts, const uint8_t* protect_opt,
                              const RowStreams* rows, float* scores_out, int32_t* keep_idx_out, int32_t* cu_keep_out, unsigned char* ws,
                              int32_t* device_status, cudaStream_t st, bool* gathered);

// Diagnostic launch counter (fastav_kernel_launches).
void count_launches(int n);

// The driver's tensor-map encoder (cuTensorMapEncodeTiled), looked up once through the runtime; nullptr if absent.
void* tensor_map_encode_entry();
// A [rows, heads, d] bf16 tensor with element strides (st, sh, 1) as a rank-3 tensor map (d, heads, rows) with the 128-byte swizzle; a
// box is a 64-element (128-byte) column block of `box_heads` heads of `box_rows` consecutive rows.  `map`: a CUtensorMap.
bool encode_rows_map(const void* ptr, int dim, int heads, long long rows, long long st, long long sh, int box_heads, int box_rows, void* map);

// A number for the calling thread's current context, never given to another one in this process; 0 if there is none (yet).
unsigned long long current_context();

__host__ __device__ inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// ---- programmatic dependent launch ----------------------------------------------------------------
// The kernels of one prune call form a chain in which each reads what its predecessor wrote.  They
// are launched with programmatic stream serialization: a kernel lets its successor start before its own end
// (pdl_trigger) so that the successor's launch and set-up overlap this kernel's tail, and every
// block of the successor calls pdl_wait -- which returns once the predecessor has completed and its
// writes are visible -- before it touches global memory another kernel may have written, or writes
// global memory another kernel may still read.  Every block waits before it exits, so completion of a
// kernel implies completion of all its predecessors.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// A pointer to data the predecessor writes must be passed through this after pdl_wait: the compiler
// may otherwise hoist loads through a `const __restrict__` pointer above the wait (it is entitled to
// assume nobody writes such data while the kernel runs).
#define pdl_acquire(ptr) asm volatile("" : "+l"(ptr) : : "memory")
// ... and must never be read through the non-coherent path (ld.global.nc, which __ldg forces): such a load can
// be served from a line this SM cached during an earlier launch, before the predecessor rewrote it (seen with a
// kernel that started early under programmatic launch and re-read a buffer of the previous call).  chain_load
// reads through L2.
template <typename T>
__device__ __forceinline__ T chain_load(const T* p) { return __ldcg(p); }
// The same for values read many times (a table that is searched): an ordinary coherent load that may stay in L1,
// spelled out so that it can never turn into the non-coherent form.
template <typename T>
__device__ __forceinline__ T chain_load_cached(const T* p) { return __ldca(p); }


// Sequence b of a packed batch as the device sees it in a prefix-sum array, cut down to what the host scalars
// promise: buffers and grids are sized from total_tokens / max_seqlen (total_q / max_qlen), loop bounds come from
// the device array, and a caller whose two views disagree must get a status bit, not an out-of-bounds access.
struct Span {
  int first, count;
  bool bad;  // the array and the host scalars disagree: the span was clamped (FASTAV_DEV_SHAPE_MISMATCH)
};
__device__ __forceinline__ Span checked_words(int a, int e, int total, int max_count) {  // of two consecutive prefix sums
  Span sp{a, e - a, false};
  if (a < 0 || a > total) {
    sp = Span{0, 0, true};
  } else {
    const int room = min(max_count, total - a);
    if (sp.count < 0) { sp.count = 0; sp.bad = true; }
    else if (sp.count > room) { sp.count = room; sp.bad = true; }
  }
  return sp;
}
// CACHED: the loads may stay in L1.  Only after the kernel's own wait (see below), and then worth it where thousands of
// blocks read the same few words: through L2 alone they queue at one slice (32 sequences, 28,672 warps: 22 us instead of 11).
template <bool CACHED = false>
__device__ __forceinline__ Span checked_span(const int32_t* cu, int b, int total, int max_count) {
  return checked_words(CACHED ? chain_load_cached(cu + b) : chain_load(cu + b), CACHED ? chain_load_cached(cu + b + 1) : chain_load(cu + b + 1),
                       total, max_count);
}
template <bool CACHED = false>
__device__ __forceinline__ Span seq_span(const Shapes& s, const int32_t* cu_seqlens, int b) {
  return checked_span<CACHED>(cu_seqlens, b, s.total_tokens, s.max_seqlen);
}
template <bool CACHED = false>
__device__ __forceinline__ Span row_span(const Shapes& s, const int32_t* cu_qlens, int b) {
  return checked_span<CACHED>(cu_qlens, b, s.total_q, s.max_qlen);
}

// The sums over the partials of TOKENS tokens `step` apart of which `have` exist: (KV head, row chunk) in that order, `most_chunks` rows
// of `stride` floats per KV head of which `chunks` hold something.  UNROLL loads in flight per token, one running sum: whoever adds them up
// gets the same bits.
template <int UNROLL, int TOKENS>
__device__ __forceinline__ void sum_of_partials(const float* col, int step, int have, int hkv, int chunks, int most_chunks, int stride, float (&total)[TOKENS]) {
  const int terms = hkv * chunks;
#pragma unroll
  for (int t = 0; t < TOKENS; ++t) total[t] = 0.f;
  int g = 0, rc = 0;  // of the next term, stepped along instead of divided out
  for (int i0 = 0; i0 < terms; i0 += UNROLL) {
    float v[UNROLL][TOKENS];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const float* const row = col + (long long)(g * most_chunks + rc) * stride;
#pragma unroll
      for (int t = 0; t < TOKENS; ++t) v[u][t] = i0 + u < terms && t < have ? chain_load(row + t * step) : 0.f;
      if (++rc == chunks) { rc = 0; ++g; }
    }
#pragma unroll
    for (int u = 0; u < UNROLL; ++u)
#pragma unroll
      for (int t = 0; t < TOKENS; ++t) total[t] += v[u][t];
  }
}
template <int UNROLL>
__device__ __forceinline__ float sum_of_partials(const float* col, int hkv, int chunks, int most_chunks, int stride) {
  float total[1];
  sum_of_partials<UNROLL>(col, 0, 1, hkv, chunks, most_chunks, stride, total);
  return total[0];
}

// Kernels read the caller's index arrays (cu_seqlens, cu_qlens, q_idx, keep_counts, protect) before their wait, and
// those may be what earlier work on the stream wrote (the cu_keep of the call before).  So the FIRST kernel an entry
// point launches waits at its very first instruction and lets its successor start only after that (chain_enter):
// whatever any kernel of the call then reads early is final.  It is launched programmatically all the same: its blocks
// are resident when the earlier work ends, which takes the launch latency out of the call (a positional prune of 8 x
// 2,230 tokens: 29.9 -> 26.4 us among others of its kind).  Under FASTAV_CHAIN_CALLS the caller vouches for those arrays
// and the first kernel is like any other.  chain_begin() marks the start of a call (per host thread).  Reads ahead of a
// kernel's own wait go through L2 (chain_load): a kernel that started while an earlier call was still running may find
// that call's lines in its L1.
//
// The arrays a kernel reads after chain_enter are named in the call: the compiler may otherwise hoist a load through a
// `const __restrict__` pointer above the wait (see pdl_acquire).
template <typename P>
__device__ __forceinline__ void chain_acquire_one(P& p) { pdl_acquire(p); }
template <typename Head, typename... P>
__device__ __forceinline__ void chain_enter(const Head& head, P&... arrays) {
  if (head.head_wait) pdl_wait();
  (chain_acquire_one(arrays), ...);
  pdl_trigger();
}
// For kernels that let their successor start later (pdl_trigger in their own time): a call's first kernel does its set-up that touches no
// global memory, then comes here.  A successor that is resident beside a kernel costs it more than its launch takes where
// the kernel is a chain of short steps, or where its blocks end at different times and the successor's take the SMs in between: started
// when the last loads have been issued, or some 3 us ahead of the end, 13 fine stages from 744 tokens take 148.8 us instead of 155.6,
// 1 x 2,048 tokens 21.0 / 22.6, 4 x 16,384 288 / 292, 32 ragged sequences of up to 8,192 301 / 307.  (Later still costs launch latency:
// the 13 stages 157 with the trigger behind the selection, 160 with the compaction's at its end.)
template <typename Head, typename... P>
__device__ __forceinline__ void chain_enter_late(const Head& head, P&... arrays) {
  if (head.head_wait) pdl_wait();
  (chain_acquire_one(arrays), ...);
}
inline thread_local bool g_chain_head = true;
inline void chain_begin(uint32_t flags) { g_chain_head = (flags & FASTAV_CHAIN_CALLS) == 0; }

// Function attributes live in a context: `set` runs on the first call in each (per call site, that is per kernel).  The eight
// latest are remembered, by the number the driver gives every context once; where it gives none, `set` runs each time.
template <typename F>
cudaError_t once_per_context(F set) {
  constexpr int kKept = 8;
  static std::atomic<unsigned long long> done[kKept];
  static std::atomic<unsigned> next{0};
  const unsigned long long context = current_context();
  if (context)
    for (const auto& d : done)
      if (d.load(std::memory_order_acquire) == context) return cudaSuccess;
  const cudaError_t e = set();
  if (e == cudaSuccess && context) done[next.fetch_add(1, std::memory_order_relaxed) % kKept].store(context, std::memory_order_release);
  return e;
}

template <typename T>
inline void mark_head(T&, bool) {}
inline void mark_head(Shapes& s, bool head) { s.head_wait = head ? 1 : 0; }
inline void mark_head(ChainHead& h, bool head) { h.head_wait = head ? 1 : 0; }

// `cluster`: blocks per thread-block cluster along x (0: none).
template <typename... KArgs, typename... Args>
cudaError_t launch_chained_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, int cluster, size_t smem, cudaStream_t stream,
                                   Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 0 ? 2 : 1;
  (mark_head(args, g_chain_head), ...);
  g_chain_head = false;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args... args) {
  return launch_chained_cluster(kernel, grid, block, 0, smem, stream, args...);
}
#endif

}  // namespace fastav
