// Fused router kernel: logits = x W^T (+ b) on tcgen05 tensor cores with fp32
// accumulators in tensor memory, fed by TMA; then, straight out of tensor memory, the
// model's gating rule, top-k, and a per-expert histogram (Eqs. 2-5).  The counts go to totals that the next
// kernel of the call reads (dispatch index, planner), or the block that finishes last publishes them and, when asked,
// runs the swap planner.
//
// One block owns 128 token rows and all N = pad16(E) expert columns.
// Warp roles: warp 0 = TMA producer, warp 1 = MMA issuer for the even k-blocks (owns the
// TMEM allocation; issuer of all k-blocks where there is one), warp 18 = MMA issuer for the odd
// k-blocks, warps 2..17 = epilogue.
// With N <= 128 there are two issuers, each accumulating its own k-blocks into its own TMEM accumulator
// (columns [0, N) and [N, 2N)): waiting for a stage, four MMAs and two commits take a warp longer than
// the tensor pipe needs for narrow tiles (4096 rows x 8 columns, d = 4096: bare main loop 13.6 us with two,
// 14.9 with one).  The epilogue adds the two accumulators.  Wider tiles keep the pipe busy from one warp
// (512 cycles per k-block at N = 256; 39.3 us either way for 14 tiles, d = 7168) and need one accumulator.
// Producer and issuers run their loops with the whole warp and one elected lane for the asynchronous
// instructions.  Written as "if (lane == 0)" around the loop, counters and descriptors are per-lane
// values that every such instruction has to fetch first: the loads of 4096 rows, d = 4096, took 17.3
// instead of 12.2 us, with the MMAs 22.1 instead of 13.6.
// Epilogue warps:  A warp may only read the 32 TMEM lanes (token rows) selected
// by warp_id % 4, so the 16 epilogue warps form 4 "row quarters" x 4 "subs"; the subs of
// a quarter split the expert columns between them in 32-column chunks, one thread per
// token row, and sub 0 writes the results.
//
// This kernel serves calls whose tile pairs fit on the GPU at once and need all of it, with gates that
// the ranking selection handles (ranking_gate).  Fewer tiles, and other gates, run fb_router_rows_kernel;
// more tiles run fb_router_persistent_kernel.
//
// Epilogue outline (after the accumulator is complete the pipeline's shared memory is
// idle and is reused as scratch):
//   pass 1  TMEM -> registers, 32 independent columns at a time: logit (+bias), selection
//           key (logit, or sigmoid + bias); keys are parked in shared memory, each chunk's best keys
//           (sigmoid gate: the group's score) in tables beside them.
//   choose  every thread picks its row's best groups and a lower bound for the k-th key.
//   pass 2  the keys that reach the bound are compacted into a list per row and ranked there.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "fb_dispatch.cuh"
#include "fb_planner.cuh"
#include "fb_ptx.cuh"

namespace fb {

constexpr int kTileM = 128;            // token rows per block
constexpr int kBlockK = 64;            // bf16 elements per k-block = one 128-byte swizzled row
constexpr int kUmmaK = 16;             // K of one tcgen05.mma for 16-bit inputs
constexpr int kMaxStages = 8;
constexpr int kEpiSubs = 4;            // epilogue warps per row quarter
constexpr int kEpilogueThreads = 128 * kEpiSubs;
constexpr int kEpilogueWarps = kEpilogueThreads / 32;
constexpr int kRouterThreads = 64 + kEpilogueThreads + 32;
constexpr int kSecondIssuerWarp = kRouterThreads / 32 - 1;
constexpr int kATileBytes = kTileM * kBlockK * 2;
constexpr int kMaxPieces = 8;                // block pairs that share a tile pair: clusters of 16 blocks
constexpr uint32_t kAccumBarrierId = 2;      // named barrier: accumulator finished (MMA warp -> epilogue warps)
constexpr uint32_t kRowBarrierBase = 3;      // named barriers 3..6: the kEpiSubs warps that share one quarter of the rows

enum RouterMode : int {
  kModePredict = 0,        // histogram -> counts
  kModePredictPlan = 1,    // histogram -> totals for the planner kernel, or -> counts -> planner in the pair that finishes last
  kModeDispatch = 2,       // ids, weights, per-tile histogram for the dispatch index
  kModeLayer = 3           // one launch for a whole layer: the first tiles_first tiles are the early pass
                           // (mode 1) on the first input, the others the normal pass (mode 2) on the
                           // second - all at the same time where every block has one tile, otherwise a
                           // block's tiles of the early pass come first
};

struct RouterParams {
  int32_t T, d, E, N, k;
  int32_t gate, n_group, topk_group, renorm;
  float route_scale;
  int32_t num_kb;                    // ceil(d / 64)
  int32_t stages;
  int32_t prefetch_kb;               // k-blocks of x that a block brings into L2 while it waits, at most (prefetch_operands)
  int32_t tmem_cols;                 // power of two >= 32 that holds acc_sets sets of N columns per issuer
  int32_t issuers;                   // MMA issuers, each with an accumulator of its own (see above)
  int32_t acc_sets;                  // sets of accumulators: 2 where a pair walks several tiles
  int32_t mode;
  int32_t tiles_first;               // kModeLayer: blocks below this index (even) belong to the early pass
  int32_t ticket_target;             // number of tickets taken: one per block that publishes counts (persistent kernel: per pair)
  int32_t fuse_planner;              // prediction modes: the block that finishes last runs the planner
  int32_t defer_counts;              // the early pass adds its counts to counts_scratch and leaves the count vector and the
                                     // plan to the next kernel: the dispatch index (kModeLayer, fb_dispatch_kernel<true>)
                                     // or the planner kernel (kModePredictPlan)
  // fb_router_rows_kernel only: J block pairs per tile pair (cluster size / 2), the rows staged at a time
  // while the operand ring is busy with the next tile, and the column layout of a row over the lanes of a
  // warp: lane l holds columns g group_size + (l % lanes_per_group) cols_per_lane + j of group
  // g = l / lanes_per_group.  Gates that keep every group have groups == 1.
  int32_t pieces, chunk_rows;
  int32_t groups, group_size, keep_groups, lanes_per_group, cols_per_lane;
  int32_t two_vectors;               // eight columns per lane, staged as two vectors 128 words apart
  int32_t vector_load;               // a lane's columns are all inside or all outside its group, and contiguous words
  int32_t ragged;                    // some lane holds fewer columns than the kernel instance is made for
  const float* logit_bias;           // [E] or nullptr
  const float* select_bias;          // [E] or nullptr
  uint32_t* counts_scratch;          // [E] the early pass's counts, zero on entry; zero again on exit, or left to the next
                                     // kernel of the call (defer_counts)
  uint32_t* ticket;                  // zero on entry, zero again on exit
  int32_t* status;
  uint32_t* counts_out;              // [E]           (predict modes)
  int32_t* topk_ids;                 // [T][k] or nullptr
  float* topk_w;                     // [T][k] or nullptr
  float* logits;                     // [T][E] or nullptr
  int32_t* early_ids;                // kModeLayer: the early pass's ids and logits, or nullptr
  float* early_logits;
  uint8_t* slice_counts;             // [tiles * pieces][slice_row_bytes(E)] (dispatch mode)
  uint32_t* totals;                  // [E] sums of that table over all slices, zero on entry (dispatch mode)
  unsigned long long* stamps;        // [blocks][64] phase time stamps (FB_TIMING builds) or nullptr
  int32_t probe;                     // measurement aid: 1 = operands are loaded but no MMA is issued and nothing
                                     // follows the main loop; 2 = with the MMAs, still nothing after them
  PlanParams plan;
};

struct TopK {
  float v[FB_MAX_TOPK];
  int32_t i[FB_MAX_TOPK];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int j = 0; j < FB_MAX_TOPK; ++j) { v[j] = -INFINITY; i[j] = 0; }
  }
  // Candidates arrive in ascending id order, so a strict comparison keeps the lower
  // id ahead of an equal key.
  __device__ __forceinline__ void insert(float x, int32_t id) {
    if (x > v[FB_MAX_TOPK - 1]) {
#pragma unroll
      for (int j = FB_MAX_TOPK - 1; j > 0; --j) {
        const bool above_prev = x > v[j - 1];
        const bool above_cur = x > v[j];
        v[j] = above_prev ? v[j - 1] : (above_cur ? x : v[j]);
        i[j] = above_prev ? i[j - 1] : (above_cur ? id : i[j]);
      }
      if (x > v[0]) { v[0] = x; i[0] = id; }
    }
  }
  // Same list, candidates in any order: equal keys are ordered by ascending id.
  __device__ __forceinline__ void insert_any_order(float x, int32_t id) {
    const bool enters = x > v[FB_MAX_TOPK - 1] || (x == v[FB_MAX_TOPK - 1] && id < i[FB_MAX_TOPK - 1]);
    if (enters) {
#pragma unroll
      for (int j = FB_MAX_TOPK - 1; j > 0; --j) {
        const bool above_prev = x > v[j - 1] || (x == v[j - 1] && id < i[j - 1]);
        const bool above_cur = x > v[j] || (x == v[j] && id < i[j]);
        v[j] = above_prev ? v[j - 1] : (above_cur ? x : v[j]);
        i[j] = above_prev ? i[j - 1] : (above_cur ? id : i[j]);
      }
      if (x > v[0] || (x == v[0] && id < i[0])) { v[0] = x; i[0] = id; }
    }
  }
};

// 1 / (1 + 2^(-z log2 e)) with the two hardware approximations (relative error ~1e-7).
// 2^x overflows to +inf for z < -88 and the reciprocal of +inf is 0, as it should be.
__device__ __forceinline__ float fb_sigmoid(float z) {
  float e, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(z * -1.4426950408889634f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + e));
  return r;
}

// Shared-memory scratch of the epilogue (it reuses the pipeline stages): keys [N][128], three tables of
// known keys per row (group scores and bounds), candidate lists.
constexpr int kCandCap = 32;           // candidates per row the fast selection path can hold
constexpr int kBoundRows = 8;          // chunks per row on that path, at most (rows of the bound tables)
__host__ __device__ constexpr size_t epilogue_scratch_bytes(int N) {
  return (static_cast<size_t>(N) * kTileM + 3 * kBoundRows * kTileM + 2 * kCandCap * kTileM) * 4;
}

// Gates that the ranking selection serves: DeepSeek-V3-like sigmoid gates (groups of exactly one
// 32-column chunk, at most 8 groups, at most kEpiSubs kept, two known keys per kept group >= k) and
// softmax gates over whole chunks (every chunk counts as a kept group; not when the softmax denominator
// is needed, i.e. weights without renormalisation).  Everything else runs fb_router_rows_kernel.
__host__ __device__ inline bool ranking_gate(int E, int k, int gate, int n_group, int topk_group, bool want_sum) {
  if (gate != FB_GATE_SOFTMAX_TOPK)
    return E / n_group == 32 && E % n_group == 0 && n_group <= 8 && topk_group <= kEpiSubs && topk_group * 2 >= k;
  return E % 32 == 0 && E / 32 <= kBoundRows && (E / 32) * 2 >= k && !want_sum;
}

// A group's score from its two best keys.  A sum that is no number counts as -inf: the ranks of the scores are then a
// permutation for every row, so that each of the best topk_group ranks has exactly one group - the warps that scan one
// group per row go through their collective steps together whatever the rows hold.
__device__ __forceinline__ float group_score(float best, float second) { return fmaxf(best + second, -INFINITY); }

struct RouterShared {
  uint64_t full_bar[kMaxStages];
  uint64_t empty_bar[kMaxStages];
  uint64_t accum_bar;
  uint32_t tmem_base;
  int32_t abort_flag;
  int32_t is_last;
  int32_t accum_ok;
  int32_t started;                           // the wait for the kernels before this one is over (prefetch_operands)
  int32_t issuer_progress[2];                // where both issuers use a stage: see issuer_turn_wait
  float logit_bias[FB_MAX_EXPERTS];
  alignas(16) float select_bias[FB_MAX_EXPERTS];
  alignas(16) uint32_t hist[FB_MAX_EXPERTS];
  uint32_t cand_count[kTileM];               // fast selection path: candidates claimed per row
  PlanShared plan;
};

// Order-preserving map of a float onto unsigned integers, and back.
__device__ __forceinline__ uint32_t ordered_bits(float x) {
  const uint32_t b = __float_as_uint(x);
  return b ^ ((b >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float from_ordered_bits(uint32_t u) {
  return __uint_as_float(u ^ ((u >> 31) ? 0x80000000u : 0xffffffffu));
}

// Sorted merge of two descending lists of three (Batcher's odd-even merge of 4 + 4 without the padding).
__device__ __forceinline__ void merge3(const float (&a)[3], const float (&b)[3], float (&o)[6]) {
  // even places a0 a2 | b0 b2 and odd places a1 | b1 merged, then neighbours compared
  const float e0 = fmaxf(a[0], b[0]), x = fminf(a[0], b[0]), y = fmaxf(a[2], b[2]), e3 = fminf(a[2], b[2]);
  const float e1 = fmaxf(x, y), e2 = fminf(x, y);
  const float d0 = fmaxf(a[1], b[1]), d1 = fminf(a[1], b[1]);
  o[0] = e0;
  o[1] = fmaxf(d0, e1); o[2] = fminf(d0, e1);
  o[3] = fmaxf(d1, e2); o[4] = fminf(d1, e2);
  o[5] = e3;
}
// The k-th largest of two descending lists: the best of "the i-th of one and the (k - i)-th of the other".
template <int kLen, int kK>
__device__ __forceinline__ float kth_of_two(const float (&a)[kLen], const float (&b)[kLen]) {
  float best = -INFINITY;
#pragma unroll
  for (int i = 0; i <= kK; ++i) {
    if (i <= kLen && kK - i <= kLen) {
      const float x = i > 0 ? a[i > 0 ? i - 1 : 0] : INFINITY, y = kK - i > 0 ? b[kK - i > 0 ? kK - i - 1 : 0] : INFINITY;
      best = fmaxf(best, fminf(x, y));
    }
  }
  return best;
}
template <int kLen>
__device__ __forceinline__ float kth_of_two(const float (&a)[kLen], const float (&b)[kLen], int k) {
  switch (k) {                                               // (the same for the whole launch)
    case 1: return kth_of_two<kLen, 1>(a, b);
    case 2: return kth_of_two<kLen, 2>(a, b);
    case 3: return kth_of_two<kLen, 3>(a, b);
    case 4: return kth_of_two<kLen, 4>(a, b);
    case 5: return kth_of_two<kLen, 5>(a, b);
    case 6: return kth_of_two<kLen, 6>(a, b);
    case 7: return kth_of_two<kLen, 7>(a, b);
    default: return kth_of_two<kLen, 8>(a, b);
  }
}
// The 8 largest of two descending lists of six, in descending order: the larger halves of a bitonic sequence
// of 16 (six and six with two -inf behind each), then a bitonic sort of 8.
__device__ __forceinline__ void merge6_top8(const float (&a)[6], const float (&b)[6], float (&o)[8]) {
  o[0] = a[0]; o[1] = a[1];
#pragma unroll
  for (int i = 2; i < 6; ++i) o[i] = fmaxf(a[i], b[7 - i]);
  o[6] = b[1]; o[7] = b[0];
#pragma unroll
  for (int w = 4; w >= 1; w >>= 1) {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if ((i & w) == 0) {
        const float hi = fmaxf(o[i], o[i + w]);
        o[i + w] = fminf(o[i], o[i + w]);
        o[i] = hi;
      }
  }
}

// The k-th largest of the known keys of a row: tab holds three tables of kBoundRows rows
// (each chunk's best, second and third key), of which the first n_chunks rows are valid
// (3 n_chunks >= k).  By merging the sorted triples (counting for every value how many are at least as
// large took 0.9 us more of a launch of one tile per pair at 4 chunks; layer step 8192 x 128 30.0 -> 28.7 us,
// 131072 x 128 211 -> 204).
__device__ __forceinline__ float kth_largest_known(const float* tab, int n_chunks, int k, int row_in_tile) {
  auto triple = [&](int c, float (&v)[3]) {
#pragma unroll
    for (int t = 0; t < 3; ++t) v[t] = c < n_chunks ? tab[(t * kBoundRows + c) * kTileM + row_in_tile] : -INFINITY;
  };
  auto six = [&](int c, float (&o)[6]) {
    float a[3], b[3];
    triple(c, a);
    triple(c + 1, b);
    merge3(a, b, o);
  };
  float p[6], q[6];
  six(0, p);
  six(2, q);
  if (n_chunks <= 4) return kth_of_two<6>(p, q, k);
  float left[8], right[8];
  merge6_top8(p, q, left);
  six(4, p);
  six(6, q);
  merge6_top8(p, q, right);
  return kth_of_two<8>(left, right, k);
}

// Ranking selection, shared by both router kernels.  cand[c * 128 + row] holds candidate c of
// the row as one 64-bit word: ordered key bits in the high half, ~expert id in the low half,
// so that "larger word" means "larger key, then lower id".  The kEpiSubs threads of a row
// share the candidates (candidate c belongs to thread c % kEpiSubs); a candidate with fewer
// than FB_MAX_TOPK larger ones is written to out_hi/out_lo[rank][row].  Returns true when
// the row had more candidates than the list holds (nothing is written for it then).
// A thread ranks kMine candidates at a time, from c0 on.  (Always four: a warp whose longest list has a
// candidate or two more than 16 went through twice the comparisons.)
template <int kMine>
__device__ __forceinline__ void rank_some(const unsigned long long* cand, uint32_t n, uint32_t n_most, uint32_t c0, int sub,
                                          int row_in_tile, uint32_t* out_hi, uint32_t* out_lo) {
  unsigned long long mykey[kMine];
  uint32_t rank[kMine];
#pragma unroll
  for (int t = 0; t < kMine; ++t) {
    const uint32_t c = c0 + t * kEpiSubs + sub;
    mykey[t] = cand[(c < n ? c : 0) * kTileM + row_in_tile];
    rank[t] = 0;
  }
#pragma unroll 2
  for (uint32_t d = 0; d < n_most; ++d) {
    const unsigned long long other = d < n ? cand[d * kTileM + row_in_tile] : 0ull;
#pragma unroll
    for (int t = 0; t < kMine; ++t) rank[t] += other > mykey[t] ? 1u : 0u;
  }
#pragma unroll
  for (int t = 0; t < kMine; ++t) {
    const uint32_t c = c0 + t * kEpiSubs + sub;
    if (c < n && rank[t] < static_cast<uint32_t>(FB_MAX_TOPK)) {
      out_hi[rank[t] * kTileM + row_in_tile] = static_cast<uint32_t>(mykey[t] >> 32);
      out_lo[rank[t] * kTileM + row_in_tile] = static_cast<uint32_t>(mykey[t]);
    }
  }
}
__device__ __forceinline__ bool rank_candidates(const unsigned long long* cand, uint32_t n_all, int sub,
                                                int row_in_tile, uint32_t* out_hi, uint32_t* out_lo) {
  const bool overflow = n_all > kCandCap;
  const uint32_t n = overflow ? 0u : n_all;
  const uint32_t n_most = __reduce_max_sync(0xffffffffu, n);
  uint32_t c0 = 0;
  if (n_most > 2 * kEpiSubs) {
    if (n_most <= 3 * kEpiSubs) {
      rank_some<3>(cand, n, n_most, 0, sub, row_in_tile, out_hi, out_lo);
      c0 = 3 * kEpiSubs;
    } else {
      rank_some<4>(cand, n, n_most, 0, sub, row_in_tile, out_hi, out_lo);
      c0 = 4 * kEpiSubs;
    }
  }
#pragma unroll 1
  for (; c0 < n_most; c0 += 2 * kEpiSubs) rank_some<2>(cand, n, n_most, c0, sub, row_in_tile, out_hi, out_lo);
  return overflow;
}

// The row's top-k list as rank_candidates left it; ranks that no candidate took hold whatever was there before
// (see fill_missing_ranks).
__device__ __forceinline__ void read_ranked(TopK& top, int k, const uint32_t* out_hi, const uint32_t* out_lo,
                                            int row_in_tile) {
#pragma unroll
  for (int j = 0; j < FB_MAX_TOPK; ++j) {
    if (j < k) {
      top.v[j] = from_ordered_bits(out_hi[j * kTileM + row_in_tile]);
      top.i[j] = static_cast<int32_t>(~out_lo[j * kTileM + row_in_tile]);
    }
  }
}

// The row's first `have` ranks are known.  Where that is fewer than k - the other keys are -inf or no numbers - the
// others get the lowest expert ids the row has not named yet: every id is below E, and as no row names an expert
// twice a tile's histogram bin stays within its byte (write_slice_counts).
__device__ __forceinline__ void fill_missing_ranks(TopK& top, uint32_t have, int k) {
  if (have >= static_cast<uint32_t>(k)) return;
  uint32_t taken = 0;
#pragma unroll
  for (int j = 0; j < FB_MAX_TOPK; ++j)
    if (j < static_cast<int>(have) && top.i[j] < FB_MAX_TOPK) taken |= 1u << top.i[j];
#pragma unroll
  for (int j = 0; j < FB_MAX_TOPK; ++j)
    if (j >= static_cast<int>(have) && j < k) {
      top.v[j] = -INFINITY;
      top.i[j] = __ffs(~taken) - 1;
      taken |= 1u << top.i[j];
    }
}
// Ranks that insertion into an empty list has taken (it takes keys above -inf only).
__device__ __forceinline__ uint32_t ranks_taken(const TopK& top) {
  uint32_t n = 0;
#pragma unroll
  for (int j = 0; j < FB_MAX_TOPK; ++j) n += top.v[j] > -INFINITY ? 1u : 0u;
  return n;
}

// Expert ids and routing weights of one token (Eq. 3's top-k with the model's weight rule).
// select_bias_s: the selection bias in shared memory.
__device__ __forceinline__ void write_row_outputs(const TopK& top, const RouterParams& p, long long row,
                                                  int32_t* out_ids, float* out_w, const float* select_bias_s) {
  const int k = p.k;
  const bool sigmoid_gate = p.gate != FB_GATE_SOFTMAX_TOPK;
#ifdef FB_DEBUG
  // what the sanitizer would catch: a chosen expert outside [0, E), a repeated expert, a row outside [0, T)
  {
    bool bad = row < 0 || row >= p.T;
#pragma unroll
    for (int j = 0; j < FB_MAX_TOPK; ++j) {
      if (j < k) {
        bad = bad || top.i[j] < 0 || top.i[j] >= p.E;
#pragma unroll
        for (int h = 0; h < FB_MAX_TOPK; ++h) bad = bad || (h < j && top.i[h] == top.i[j]);
      }
    }
    if (bad) atomicCAS(p.status, 0, FB_ERR_INTERNAL);
  }
#endif
  // 16 bytes a store where every row starts on 16 bytes (a warp's rows lie k words apart)
  const bool whole = k % 4 == 0;
  if (out_ids != nullptr) {
    if (whole && reinterpret_cast<uintptr_t>(out_ids) % 16 == 0) {
#pragma unroll
      for (int j = 0; j < FB_MAX_TOPK; j += 4)
        if (j < k) *reinterpret_cast<int4*>(out_ids + row * k + j) = make_int4(top.i[j], top.i[j + 1], top.i[j + 2], top.i[j + 3]);
    } else {
#pragma unroll
      for (int j = 0; j < FB_MAX_TOPK; ++j)
        if (j < k) out_ids[row * k + j] = top.i[j];
    }
  }
  if (out_w != nullptr) {
    float w[FB_MAX_TOPK];
    float wsum = 0.0f;
    const float ref = top.v[0];                         // row maximum of the keys
#pragma unroll
    for (int j = 0; j < FB_MAX_TOPK; ++j) {
      if (!sigmoid_gate) w[j] = (j < k) ? __expf(top.v[j] - ref) : 0.0f;
      else w[j] = (j < k) ? top.v[j] - select_bias_s[top.i[j]] : 0.0f;   // unbiased sigmoid score
      wsum += w[j];
    }
    float scale;
    if (!sigmoid_gate) scale = 1.0f / wsum;
    else scale = p.renorm ? p.route_scale / wsum : p.route_scale;
    if (whole && reinterpret_cast<uintptr_t>(out_w) % 16 == 0) {
#pragma unroll
      for (int j = 0; j < FB_MAX_TOPK; j += 4)
        if (j < k)
          *reinterpret_cast<float4*>(out_w + row * k + j) = make_float4(w[j] * scale, w[j + 1] * scale, w[j + 2] * scale, w[j + 3] * scale);
    } else {
#pragma unroll
      for (int j = 0; j < FB_MAX_TOPK; ++j)
        if (j < k) out_w[row * k + j] = w[j] * scale;
    }
  }
}

// End of a tile in the prediction modes: add the tile's histogram (shared memory, cleared
// here) to the cross-block counts, take a ticket, and in the block that takes the last one
// publish the count vector (Eq. 5), re-arm the scratch for the next call and run the planner
// (Algorithm 1) when asked.  Called by all epilogue threads; et = thread index among them.
template <class Shared>
__device__ __forceinline__ void publish_counts(Shared& sh, const RouterParams& p, int et, int warp, int lane,
                                               bool run_planner) {
  for (int e = et; e < p.E; e += kEpilogueThreads) {
    const uint32_t c = sh.hist[e];
    if (c) atomicAdd(&p.counts_scratch[e], c);
    sh.hist[e] = 0;
  }
  named_bar_sync(kPlanBarrierId, kEpilogueThreads);
  if (et == 0) {
    // The barrier orders every thread's histogram atomics before this fence, and the
    // fence (cumulative) publishes them device-wide before the ticket is taken.
    fence_acq_rel_gpu();
    const uint32_t prev = atomicAdd(p.ticket, 1u);
    const bool last = prev == static_cast<uint32_t>(p.ticket_target) - 1;
    // Acquire side of the same hand-shake: the other blocks' counts are visible to this thread
    // after the fence and, through the barrier below, to the whole block.
    if (last) fence_acq_rel_gpu();
    sh.is_last = last ? 1 : 0;
  }
  named_bar_sync(kPlanBarrierId, kEpilogueThreads);
  FB_STAMP(11, 64);
  if (sh.is_last) {
    // Every other tile has published its counts: this block finishes the pass.
    for (int e = et; e < p.E; e += kEpilogueThreads) {
      const uint32_t c = __ldcg(&p.counts_scratch[e]);
      p.counts_out[e] = c;
      if (run_planner) plan_put_count(sh.plan, e, c);
      p.counts_scratch[e] = 0;           // ready for the next call
    }
    if (et == 0) *p.ticket = 0;
    if (sh.abort_flag) { if (et == 0) atomicCAS(p.status, 0, FB_ERR_TIMEOUT); }
    if (run_planner) {
      named_bar_sync(kPlanBarrierId, kEpilogueThreads);
      if (warp == 2)
        plan_swaps_apart(p.plan, sh.plan, lane, p.status,
                         p.stamps != nullptr ? p.stamps + static_cast<size_t>(blockIdx.x) * 64 : nullptr);
      named_bar_sync(kPlanBarrierId, kEpilogueThreads);
      plan_write_placement(p.plan, sh.plan, et, kEpilogueThreads);
    }
  }
}

// A tile's histogram as one table row of the dispatch index: one byte per expert (a count is at most
// kTileM), four per store.  Bins from E up to the row's end are zero.
__device__ __forceinline__ void write_slice_counts(uint8_t* table, int slice, int E, const uint32_t* hist, int et) {
  const int row_bytes = slice_row_bytes(E);
  for (int w = et; w < row_bytes / 4; w += kEpilogueThreads) {
    const uint4 h = *reinterpret_cast<const uint4*>(hist + 4 * w);
    reinterpret_cast<uint32_t*>(table + static_cast<size_t>(slice) * row_bytes)[w] =
        h.x | h.y << 8 | h.z << 16 | h.w << 24;
  }
}

// A block's counts into the sums over all blocks that the dispatch-index kernel reads: thread et adds expert et's.
// Nothing here waits for the additions, the end of the grid does.
__device__ __forceinline__ void add_to_totals(uint32_t* totals, int E, uint32_t count, int et) {
  static_assert(kEpilogueThreads >= FB_MAX_EXPERTS, "one thread per expert");
  if (et < E && count != 0) atomicAdd(totals + et, count);
}

// Two MMA issuers share one ring of stages.  Where a stage always serves the same issuer - an even number of stages, and
// one tile per pair or an even number of k-blocks per tile - that issuer sees every phase of the stage's "full" barrier.
// With an odd number of stages a stage alternates between them, and with an odd number of k-blocks the issuers' ring
// positions trade places from tile to tile; a parity wait alone cannot tell "the other issuer's use of this stage is
// still being filled" (a wait for my parity passes on the phase before it) from "my use is complete".  So each issuer
// publishes the ring position of the last k-block whose operands it has seen arrive, and before it waits for position g on
// a stage whose previous use (position g - stages) was the other issuer's, it waits until the other one has got that far.
__device__ __forceinline__ bool issuer_turn_wait(const volatile int32_t* other_progress, int32_t need,
                                                 volatile int* abort_flag) {
  uint32_t polls = 0;
  uint64_t t0 = 0;
  while (*other_progress < need) {
    if ((++polls & 0x3Fu) == 0) {
      if (*abort_flag) return false;
      const uint64_t now = global_timer_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > kWaitLimitNs) { *abort_flag = 1; return false; }
    }
  }
  return true;
}

__device__ __forceinline__ void ring_advance(int& s, uint32_t& phase, int stages) {
  if (++s == stages) { s = 0; phase ^= 1u; }
}

// The tile pairs of a block pair and its share of their k-blocks: pair_first, pair_first + pair_stride, ...;
// in kModeLayer the first pairs_per_pass pairs belong to the early pass, the rest to the normal pass.
struct TileWalk {
  int pair_first, pair_stride, total_pairs, pairs_per_pass;
  int kb0, n_kb;
  uint32_t cluster_rank;
};

// While a block waits for the stream's earlier kernels (blocks start as soon as SMs are free) its second issuer warp brings
// the first of its rows of x into L2.  Nothing is read early: L2 is where this GPU's writes meet its reads, so a line
// that an earlier kernel still writes is written there and read after the wait.  Memory is idle meanwhile where the kernel
// before is a dispatch index or a planner: layer calls back to back without and with it, 8192 tokens x 2048, 128 experts 23.8
// and 22.4 us, 4096 x 4096, 8 experts 20.1 and 18.7, prediction and plan of 8192 x 2048 17.1 and 16.2.  Behind a kernel that
// does not let this one start early there is nothing to gain: 24.0 and 24.7, 21.2 and 21.2, 17.3 and 17.3.
// After as many k-blocks as the ring holds, one every kPrefetchCycles - an SM's share of the memory bandwidth - so that the
// loads that follow the wait never queue behind many of these; the limit on all blocks' together (prefetch_kb) keeps
// what is brought in well inside the 126 MB of L2.
constexpr int kPrefetchCycles = 600;
constexpr int kPrefetchBytes = 48 << 20;
__device__ __forceinline__ void prefetch_operands(const RouterParams& p, const CUtensorMap* map_x, const CUtensorMap* map_x2,
                                                  const TileWalk& w, const volatile int32_t* started) {
  const bool leader = elect_one();
  int n = 0;
  for (int pt = w.pair_first; pt < w.total_pairs && n < p.prefetch_kb; pt += w.pair_stride) {
    const bool second_pass = pt >= w.pairs_per_pass;
    const int row = (2 * (second_pass ? pt - w.pairs_per_pass : pt) + static_cast<int>(w.cluster_rank & 1u)) * kTileM;
    const CUtensorMap* xmap = second_pass ? map_x2 : map_x;
    for (int kb = w.kb0; kb < w.kb0 + w.n_kb && n < p.prefetch_kb && row < p.T; ++kb, ++n) {
      const long long t0 = clock64();
      do {
        if (*started) return;
      } while (n >= p.stages && clock64() - t0 < kPrefetchCycles);
      if (leader) tma_prefetch_2d(xmap, kb * kBlockK, row);
    }
  }
}

// L2 policies of the operand loads.  x is streamed once - unless the logits are written as well: who asks for them compares
// the two passes and reads the hidden states again (call and quality figures, 8192 x 2048, 128 experts: 49.7 -> 47.7 us).  W is
// re-read by every pair.  Made by the producer warp before its wait for the stream's earlier kernels: behind the wait the choice
// between the two took 0.1 us of every launch (8 experts, 128 tokens, prediction 7.00 -> 7.09 us).
struct LoadPolicies { uint64_t x, w; };
__device__ __forceinline__ LoadPolicies load_policies(const RouterParams& p) {
  return {p.logits != nullptr ? l2_policy_evict_normal() : l2_policy_evict_first(), l2_policy_evict_last()};
}

// TMA producer (a whole warp): both blocks of a pair report their bytes to the even block's barrier, which
// expects the bytes of both.
__device__ __forceinline__ void produce_operands(const RouterParams& p, const CUtensorMap* map_x, const CUtensorMap* map_x2,
                                                 const CUtensorMap* map_w, const TileWalk& w, uint32_t smem_base,
                                                 uint32_t stage_bytes, uint64_t* full_bar, uint64_t* empty_bar,
                                                 const LoadPolicies& policy, volatile int* abort_flag) {
  const bool leader = elect_one();
  const uint32_t cta_rank = w.cluster_rank & 1u;
  const int stages = p.stages, w_row = static_cast<int>(cta_rank) * (p.N / 2);
  int s = 0;
  uint32_t phase = 0;
  bool ok = true;
  for (int pt = w.pair_first; pt < w.total_pairs && ok; pt += w.pair_stride) {
    const bool second_pass = pt >= w.pairs_per_pass;
    const int row = (2 * (second_pass ? pt - w.pairs_per_pass : pt) + static_cast<int>(cta_rank)) * kTileM;
    const CUtensorMap* xmap = second_pass ? map_x2 : map_x;
    for (int kb = w.kb0; kb < w.kb0 + w.n_kb; ++kb) {
      ok = __all_sync(0xffffffffu, mbar_wait<true>(smem_u32(&empty_bar[s]), phase ^ 1u, abort_flag));
      if (!ok) break;
      if (kb == w.kb0) FB_STAMP(14, 0);
      if (kb == w.kb0 + w.n_kb - 1) FB_STAMP(15, 0);
      if (leader) {
        const uint32_t a_dst = smem_base + static_cast<uint32_t>(s) * stage_bytes;
        const uint32_t full = map_to_cta(smem_u32(&full_bar[s]), w.cluster_rank & ~1u);
        if (cta_rank == 0) mbar_arrive_expect_tx(smem_u32(&full_bar[s]), 2u * stage_bytes);
        tma_load_2d_pair(a_dst, xmap, full, kb * kBlockK, row, policy.x);
        tma_load_2d_pair(a_dst + kATileBytes, map_w, full, kb * kBlockK, w_row, policy.w);
      }
      __syncwarp();
      ring_advance(s, phase, stages);
    }
  }
}

// MMA issuer (a whole warp of the pair's even block): issuer 0 takes the k-blocks 0, 2, 4, ... of every
// tile, issuer 1 the others; a single issuer takes all.  accum_bar[set] completes when the tile is done,
// tmem_empty_bar[set] (several tiles only) when its accumulators have been read out.
__device__ __forceinline__ void issue_mmas(const RouterParams& p, const TileWalk& w, int issuer, uint32_t tmem_base,
                                           uint32_t smem_base, uint32_t stage_bytes, uint64_t* full_bar, uint64_t* empty_bar,
                                           uint64_t* accum_bar, uint64_t* tmem_empty_bar, int32_t* progress,
                                           volatile int* abort_flag) {
  const bool leader = elect_one();
  const int stages = p.stages, step = p.issuers;
  const uint32_t idesc = umma_idesc_bf16_f32(kTileM * 2, static_cast<uint32_t>(p.N));
  const bool several = w.pair_first + w.pair_stride < w.total_pairs;
  const bool shared_stages = step == 2 && ((stages & 1) != 0 || (several && (w.n_kb & 1) != 0));   // see issuer_turn_wait
  volatile int32_t* my_progress = progress + issuer;
  const volatile int32_t* other_progress = progress + (issuer ^ 1);
  int s0 = 0;                                  // stage and phase of the tile's first k-block
  uint32_t phase0 = 0;
  int32_t g0 = 0;                              // its ring position: k-blocks of all of this pair's tiles, in order
  uint32_t set = 0, use = 0;
  bool ok = true;
  for (int pt = w.pair_first; pt < w.total_pairs && ok; pt += w.pair_stride) {
    const uint32_t acc = tmem_base + (set * static_cast<uint32_t>(step) + static_cast<uint32_t>(issuer)) * static_cast<uint32_t>(p.N);
    if (use != 0) {
      // the set's previous contents must have been read out by both blocks
      ok = __all_sync(0xffffffffu, mbar_wait<true>(smem_u32(&tmem_empty_bar[set]), (use - 1u) & 1u, abort_flag));
      if (!ok) break;
      tcgen05_fence_after();
    }
    int s = s0 + issuer;
    uint32_t phase = phase0;
    if (s >= stages) { s -= stages; phase ^= 1u; }
    for (int kb = issuer; kb < w.n_kb; kb += step) {
      if (shared_stages && g0 + kb >= stages) {
        // whose was the stage's previous use (ring position g0 + kb - stages)?  Its k-block index
        // inside its own tile decides, as for every k-block.
        int kbp = kb - stages;
        while (kbp < 0) kbp += w.n_kb;
        if ((kbp & 1) != issuer)
          ok = __all_sync(0xffffffffu, issuer_turn_wait(other_progress, g0 + kb - stages, abort_flag));
      }
      ok = ok && __all_sync(0xffffffffu, mbar_wait<true>(smem_u32(&full_bar[s]), phase, abort_flag));
      if (!ok) break;
      if (shared_stages && leader) *my_progress = g0 + kb;
      tcgen05_fence_after();
      if (kb == 0) FB_STAMP(16, 32);
      const uint32_t a_addr = smem_base + static_cast<uint32_t>(s) * stage_bytes;
      const uint64_t adesc = umma_smem_desc_sw128(a_addr);
      const uint64_t bdesc = umma_smem_desc_sw128(a_addr + kATileBytes);
      if (leader) {
        if (p.probe != 1) {
          // advance 16 elements = 32 bytes inside the swizzled row: +2 in the address field
#pragma unroll
          for (int kk = 0; kk < kBlockK / kUmmaK; ++kk)
            umma_bf16<2>(acc, adesc + 2u * kk, bdesc + 2u * kk, idesc, (kb != issuer || kk != 0) ? 1u : 0u);
        }
        umma_commit_pair(smem_u32(&empty_bar[s]), w.cluster_rank);   // frees the stage in both blocks when these retire
      }
      __syncwarp();
      s += step;
      if (s >= stages) { s -= stages; phase ^= 1u; }
    }
    if (issuer == 0) FB_STAMP(17, 32);
    if (ok && leader) umma_commit_pair(smem_u32(&accum_bar[set]), w.cluster_rank);   // this issuer's accumulator is complete
    __syncwarp();
    g0 += w.n_kb;
    s0 += w.n_kb % stages;
    phase0 ^= static_cast<uint32_t>(w.n_kb / stages) & 1u;
    if (s0 >= stages) { s0 -= stages; phase0 ^= 1u; }
    if (++set == static_cast<uint32_t>(p.acc_sets)) { set = 0; ++use; }
  }
}

// One tile pair per block pair.  Launched in clusters of two; the pair shares one 256 x N MMA
// (tcgen05 cta_group::2).  Each block loads its own 128 rows of x and half of the W tile.  The even
// block of the pair issues the MMAs and owns the "full" barriers; both blocks get their stage-free and
// accumulator-ready signals from its commits.
// kSigmoid: DeepSeek-V3-like sigmoid gate or softmax gate over whole chunks (see ranking_gate).
// kLogitBias: whether a logit bias (Eq. 2's "+ b") is given; without it the key computation
// shrinks to one variant.
template <bool kSigmoid, bool kLogitBias>
__global__ void __launch_bounds__(kRouterThreads, 1)
fb_router_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_x2,
                 const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ RouterParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ RouterShared sh;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);      // warp-uniform for the compiler as well
  const int lane = threadIdx.x & 31;
  // kModeLayer: which pass this block belongs to, its tile there and its input
  const int owner_block = static_cast<int>(blockIdx.x);
  const bool second_pass = p.mode == kModeLayer && owner_block >= p.tiles_first;
  const int mode = p.mode == kModeLayer ? (second_pass ? kModeDispatch : kModePredictPlan) : p.mode;
  const int tile = second_pass ? owner_block - p.tiles_first : owner_block;
  const bool two_acc = p.issuers == 2 && p.num_kb > 1;
  const CUtensorMap* xmap = second_pass ? &tmap_x2 : &tmap_x;
  // outputs of the normal pass are not written by blocks of the early pass
  int32_t* const out_ids = (p.mode == kModeLayer && !second_pass) ? p.early_ids : p.topk_ids;
  float* const out_logits = (p.mode == kModeLayer && !second_pass) ? p.early_logits : p.logits;
  float* const out_w = (p.mode == kModeLayer && !second_pass) ? nullptr : p.topk_w;
  const uint32_t cta_rank = cluster_ctarank();
  const uint32_t b_tile_bytes = static_cast<uint32_t>(p.N / 2) * kBlockK * 2;
  const uint32_t stage_bytes = kATileBytes + b_tile_bytes;
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;   // swizzle atoms need 1024-byte alignment
  volatile int* abort_flag = &sh.abort_flag;
  FB_STAMP(0, 64);

  if (threadIdx.x == 0) {
    sh.abort_flag = 0;
    sh.is_last = 0;
    sh.started = 0;
    sh.issuer_progress[0] = -1;
    sh.issuer_progress[1] = -1;
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&sh.full_bar[s]), 1);
      mbar_init(smem_u32(&sh.empty_bar[s]), 1);
    }
    mbar_init(smem_u32(&sh.accum_bar), static_cast<uint32_t>(p.issuers));      // one commit per MMA issuer
    fence_mbar_init();
    prefetch_tensormap(xmap);
    prefetch_tensormap(&tmap_w);
  }
  if (warp == 1) {
    tmem_alloc<2>(smem_u32(&sh.tmem_base), static_cast<uint32_t>(p.tmem_cols));
    tmem_relinquish<2>();
  }
  if (warp >= 2) {
    const int et = threadIdx.x - 64;
    for (int e = et; e < FB_MAX_EXPERTS; e += kEpilogueThreads) {
      sh.hist[e] = 0;
      if (e < kTileM) sh.cand_count[e] = 0;
    }
    if (mode == kModePredictPlan && !p.defer_counts) plan_clear(sh.plan, et, kEpilogueThreads);
  }
  tcgen05_fence_before();
  __syncthreads();
  cluster_arrive_relaxed(); cluster_wait();  // the partner's barriers and TMEM are ready too
  tcgen05_fence_after();
  TileWalk walk;
  walk.pair_first = static_cast<int>(blockIdx.x) / 2;
  walk.pair_stride = walk.total_pairs = static_cast<int>(gridDim.x) / 2;       // one tile pair per block pair
  walk.pairs_per_pass = p.tiles_first / 2;
  walk.kb0 = 0;
  walk.n_kb = p.num_kb;
  walk.cluster_rank = cta_rank;
  LoadPolicies policies = {0, 0};
  if (warp == 0) policies = load_policies(p);
  if (warp == kSecondIssuerWarp) prefetch_operands(p, &tmap_x, &tmap_x2, walk, &sh.started);
  // Everything above touched only this block's own state and the call's parameters; from here on
  // the kernel reads memory that earlier work of the stream may have written.
  pdl_wait();
  if (threadIdx.x == 0) *static_cast<volatile int32_t*>(&sh.started) = 1;
  // From here on the next kernel of the stream may be scheduled (if it was launched with
  // programmatic stream serialization - the library's own router launches are): its blocks
  // take the SMs as this grid's blocks leave them and do their set-up while the last blocks
  // of this grid finish; they read nothing before their own griddepcontrol.wait, which returns
  // only when this grid has completed.  Issued after this block's wait, so a dependent never
  // starts before everything this grid itself depended on is complete.
  pdl_launch_dependents();
  const uint32_t tmem_base = sh.tmem_base;
  FB_STAMP(1, 64);

  if (warp == 0) {
    produce_operands(p, &tmap_x, &tmap_x2, &tmap_w, walk, smem_base, stage_bytes, sh.full_bar, sh.empty_bar, policies, abort_flag);
    cluster_arrive_relaxed();  // this warp is done with the pair's shared state (see the teardown)
  } else if (warp == 1 || warp == kSecondIssuerWarp) {
    // MMA issuers: in a pair only the even block issues
    if (cta_rank == 0 && (warp == 1 || p.issuers == 2))
      issue_mmas(p, walk, warp == 1 ? 0 : 1, tmem_base, smem_base, stage_bytes, sh.full_bar, sh.empty_bar, &sh.accum_bar,
                 nullptr, sh.issuer_progress, abort_flag);
    if (warp == 1) {
      // One thread polls for the finished accumulator on behalf of the 16 epilogue warps,
      // which sleep at a hardware barrier meanwhile (no issue slots, no power).
      if (lane == 0) sh.accum_ok = mbar_wait<true>(smem_u32(&sh.accum_bar), 0u, abort_flag) ? 1 : 0;
      __syncwarp();
      named_bar_arrive(kAccumBarrierId, kEpilogueThreads + 32);
    }
    __syncwarp();
    cluster_arrive_relaxed();
  } else {
    // ------------------------------------------------------------ epilogue
    const int et = threadIdx.x - 64;                       // 0 .. kEpilogueThreads-1
    const int quarter = warp & 3;                          // TMEM lanes this warp may touch
    const int sub = (warp - 2) >> 2;                       // which share of the columns
    const int row_in_tile = quarter * 32 + lane;
    const long long row = static_cast<long long>(tile) * kTileM + row_in_tile;
    const bool valid = row < p.T;
    const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
    const int E = p.E, N = p.N, k = p.k;                   // N == E: whole 32-column chunks only
    const int n_chunks = E >> 5;                           // sub s owns chunks s and s + kEpiSubs
    // While the main loop runs, stage the biases (read by these warps only, after the barrier
    // below) and the placement for the planner (any block may turn out to be the last one).
    for (int e = et; e < FB_MAX_EXPERTS; e += kEpilogueThreads) {
      sh.logit_bias[e] = (p.logit_bias != nullptr && e < p.E) ? p.logit_bias[e] : 0.0f;
      sh.select_bias[e] = (p.select_bias != nullptr && e < p.E) ? p.select_bias[e] : 0.0f;
    }
    if (mode == kModePredictPlan && !p.defer_counts) plan_load_placement(p.plan, sh.plan, et, kEpilogueThreads);
    named_bar_sync(kAccumBarrierId, kEpilogueThreads + 32);
    const bool got = sh.accum_ok != 0 && p.probe == 0;     // a measurement launch ends with its main loop
    tcgen05_fence_after();
    FB_STAMP(2, 64);

    // scratch carved out of the (now idle) pipeline stages
    float* key_s = reinterpret_cast<float*>(smem_raw + (smem_base - smem_u32(smem_raw)));   // [N][128]
    float* gscore_s = key_s + static_cast<size_t>(N) * kTileM;                               // [3 * kBoundRows][128]
    float* glow_s = gscore_s + kBoundRows * kTileM;                                          // (its second table)
    unsigned long long* cand = reinterpret_cast<unsigned long long*>(gscore_s + 3 * kBoundRows * kTileM);   // see rank_candidates
    uint32_t* out_hi = reinterpret_cast<uint32_t*>(gscore_s);               // [8][128], group scores are dead by then
    uint32_t* out_lo = out_hi + FB_MAX_TOPK * kTileM;

    // Between pass 1 and the histogram, data passes only between the kEpiSubs warps that share
    // this warp's rows: they meet at a barrier of their own and do not wait for the other rows' warps.
    auto row_sync = [&]() { named_bar_sync(kRowBarrierBase + static_cast<uint32_t>(quarter), kEpiSubs * 32); };

    if (got) {
      // ---------------- pass 1: keys of this warp's chunks, 32 columns at a time
#pragma unroll 1
      for (int c = sub; c < n_chunks; c += kEpiSubs) {
        const int c0 = c * 32;
        uint32_t r[32];
        float q[32];
        {
          // both accumulators' loads in flight at once, one wait
          uint32_t r2[32];
          tmem_ld_32x32b_x32(taddr + c0, r);
          if (two_acc) tmem_ld_32x32b_x32(taddr + N + c0, r2);
          tmem_ld_wait();
          if (two_acc) {
#pragma unroll
            for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(r2[j]));
          }
        }
        if (out_logits != nullptr && valid) {
          float4* const dst = reinterpret_cast<float4*>(out_logits + row * E + c0);
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            float4 z = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]), __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
            if (kLogitBias) {
              z.x += sh.logit_bias[c0 + j]; z.y += sh.logit_bias[c0 + j + 1];
              z.z += sh.logit_bias[c0 + j + 2]; z.w += sh.logit_bias[c0 + j + 3];
            }
            dst[j / 4] = z;
          }
        }
        if (kSigmoid && !kLogitBias) {
          // Every key goes through the same two hardware approximations, so equal logits give equal keys
          // in every column (an FMA-pipe reciprocal on alternate columns was no faster and broke exact ties).
          const float4* sb4 = reinterpret_cast<const float4*>(&sh.select_bias[c0]);
#pragma unroll
          for (int j4 = 0; j4 < 8; ++j4) {
            const float4 b = sb4[j4];
            q[4 * j4 + 0] = fb_sigmoid(__uint_as_float(r[4 * j4 + 0])) + b.x;
            q[4 * j4 + 1] = fb_sigmoid(__uint_as_float(r[4 * j4 + 1])) + b.y;
            q[4 * j4 + 2] = fb_sigmoid(__uint_as_float(r[4 * j4 + 2])) + b.z;
            q[4 * j4 + 3] = fb_sigmoid(__uint_as_float(r[4 * j4 + 3])) + b.w;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float z = __uint_as_float(r[j]) + (kLogitBias ? sh.logit_bias[c0 + j] : 0.0f);
            q[j] = kSigmoid ? fb_sigmoid(z) + sh.select_bias[c0 + j] : z;
          }
        }
        float* kcol = key_s + c0 * kTileM + row_in_tile;
#pragma unroll
        for (int j = 0; j < 32; ++j) kcol[j * kTileM] = q[j];
        if (kSigmoid) {
          // the chunk is one group: branch-free top-2 of its 32 keys by a merge tree
          float a1[16], a2[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) { a1[j] = fmaxf(q[2 * j], q[2 * j + 1]); a2[j] = fminf(q[2 * j], q[2 * j + 1]); }
#pragma unroll
          for (int w = 8; w >= 1; w >>= 1) {
#pragma unroll
            for (int j = 0; j < w; ++j) {
              const float hi = fmaxf(a1[j], a1[j + w]);
              a2[j] = fmaxf(fminf(a1[j], a1[j + w]), fmaxf(a2[j], a2[j + w]));
              a1[j] = hi;
            }
          }
          gscore_s[c * kTileM + row_in_tile] = group_score(a1[0], a2[0]);
          glow_s[c * kTileM + row_in_tile] = a2[0];
        } else {
          // the chunk's three best keys (sorted) feed the bound
          float a1[16], a2[16], a3[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            a1[j] = fmaxf(q[2 * j], q[2 * j + 1]); a2[j] = fminf(q[2 * j], q[2 * j + 1]); a3[j] = -INFINITY;
          }
#pragma unroll
          for (int w = 8; w >= 1; w >>= 1) {
#pragma unroll
            for (int j = 0; j < w; ++j) {
              // best three of two sorted triples
              const float lo1 = fminf(a1[j], a1[j + w]), hi2 = fmaxf(a2[j], a2[j + w]);
              a1[j] = fmaxf(a1[j], a1[j + w]);
              a2[j] = fmaxf(lo1, hi2);
              a3[j] = fmaxf(fminf(lo1, hi2), fmaxf(a3[j], a3[j + w]));
            }
          }
          gscore_s[c * kTileM + row_in_tile] = a1[0];
          gscore_s[(kBoundRows + c) * kTileM + row_in_tile] = a2[0];
          gscore_s[(2 * kBoundRows + c) * kTileM + row_in_tile] = a3[0];
        }
      }
    }
    FB_STAMP(3, 64);
    tcgen05_fence_before();
    // This warp has read its part of tensor memory: its share of the pair's closing barrier
    // is delivered now, so that nobody waits for it at the end (see the teardown).
    cluster_arrive_relaxed();
    row_sync();
    FB_STAMP(4, 64);
    if (got) {
      // ---------------- choose: rank the (at most 8) group scores of this row
      int my_groups[2] = {-1, -1};                        // the 32-column groups this sub scans
      float floor_key = INFINITY;
      if (kSigmoid) {
        float sc[8];
#pragma unroll
        for (int g = 0; g < 8; ++g) sc[g] = g < n_chunks ? gscore_s[g * kTileM + row_in_tile] : -INFINITY;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          int rank = 0;
#pragma unroll
          for (int h = 0; h < 8; ++h)          // a lower-numbered group wins ties
            if (h != g) rank += (h < g ? sc[h] >= sc[g] : sc[h] > sc[g]) ? 1 : 0;
          if (g < n_chunks && rank < p.topk_group) {
            floor_key = fminf(floor_key, glow_s[g * kTileM + row_in_tile]);
            if (rank == sub) my_groups[0] = g;   // sub s scans the row's s-th best group
          }
        }
      } else {
        // bound for the k-th key: the k-th largest of the chunks' three best keys (3 n_chunks >= k of them)
        floor_key = kth_largest_known(gscore_s, n_chunks, k, row_in_tile);
        if (sub < n_chunks) my_groups[0] = sub;
        if (sub + kEpiSubs < n_chunks) my_groups[1] = sub + kEpiSubs;
      }
      FB_STAMP(5, 64);
      // ---------------- collect the keys >= floor (at least k keys qualify: the bound is one of k known keys; fewer
      // only where keys are no numbers)
#pragma unroll 1
      for (int gi = 0; gi < 2; ++gi) {
        if (my_groups[gi] < 0) continue;                  // no such group: true for the whole warp at once
        const int base = my_groups[gi] * 32;              // (which group may differ from row to row)
        uint32_t mask = 0;
#pragma unroll
        for (int j = 0; j < 32; ++j)
          mask |= (key_s[(base + j) * kTileM + row_in_tile] >= floor_key) ? (1u << j) : 0u;
        const uint32_t mine = __popc(mask);
        const uint32_t first = atomicAdd(&sh.cand_count[row_in_tile], mine);
        const uint32_t most = __reduce_max_sync(0xffffffffu, mine);
#pragma unroll 1
        for (uint32_t i = 0; i < most; ++i) {
          if (mask != 0 && first + i < kCandCap) {
            const int j = __ffs(mask) - 1;
            mask &= mask - 1;
            cand[(first + i) * kTileM + row_in_tile] =
                (static_cast<unsigned long long>(ordered_bits(key_s[(base + j) * kTileM + row_in_tile])) << 32) |
                ~static_cast<uint32_t>(base + j);
          }
        }
      }
    }
    row_sync();
    FB_STAMP(7, 64);
    bool overflow = false;
    uint32_t n_cand = 0;
    if (got) {
      n_cand = sh.cand_count[row_in_tile];
      overflow = rank_candidates(cand, n_cand, sub, row_in_tile, out_hi, out_lo);
    }
    row_sync();
    FB_STAMP(8, 64);
    if (got && sub == 0) {
      TopK top;
      top.init();
      if (!overflow) read_ranked(top, k, out_hi, out_lo, row_in_tile);
      if (__any_sync(0xffffffffu, overflow || n_cand < static_cast<uint32_t>(k))) {
        // More than kCandCap keys reached the floor (many equal keys): plain scan of the
        // kept groups for the rows concerned.  Or fewer than k did (keys that are no numbers).
        if (overflow && !kSigmoid) {
          top.init();
          for (int e = 0; e < E; ++e) {
            const float x = key_s[e * kTileM + row_in_tile];
            if (x > top.v[FB_MAX_TOPK - 1]) top.insert(x, e);
          }
        } else if (overflow) {
          float sc[8];
#pragma unroll
          for (int g = 0; g < 8; ++g) sc[g] = -INFINITY;
          // group scores were overwritten by the output area: recompute them from the keys
          for (int g = 0; g < n_chunks; ++g) {
            float a1 = -INFINITY, a2 = -INFINITY;
            for (int j = 0; j < 32; ++j) {
              const float x = key_s[(g * 32 + j) * kTileM + row_in_tile];
              a2 = fmaxf(a2, fminf(a1, x));
              a1 = fmaxf(a1, x);
            }
#pragma unroll
            for (int h = 0; h < 8; ++h) if (h == g) sc[h] = group_score(a1, a2);
          }
          top.init();
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            int rank = 0;
#pragma unroll
            for (int h = 0; h < 8; ++h)
              if (h != g) rank += (h < g ? sc[h] >= sc[g] : sc[h] > sc[g]) ? 1 : 0;
            if (g < n_chunks && rank < p.topk_group) {
              for (int j = 0; j < 32; ++j) {
                const float x = key_s[(g * 32 + j) * kTileM + row_in_tile];
                if (x >= top.v[FB_MAX_TOPK - 1]) top.insert_any_order(x, g * 32 + j);
              }
            }
          }
        }
        fill_missing_ranks(top, overflow ? ranks_taken(top) : n_cand, k);
      }
      FB_STAMP(9, 64);
      if (valid) {
        // softmax gates come here with renormalised weights only: no denominator needed
        write_row_outputs(top, p, row, out_ids, out_w, sh.select_bias);
        // histogram (Eq. 5): many bins, lanes rarely collide
#pragma unroll
        for (int j = 0; j < FB_MAX_TOPK; ++j)
          if (j < k) atomicAdd(&sh.hist[top.i[j]], 1u);
      }
      FB_STAMP(10, 64);
    }
    named_bar_sync(kPlanBarrierId, kEpilogueThreads);
    if (mode == kModeDispatch || p.defer_counts) {
      if (static_cast<long long>(tile) * kTileM < p.T) {     // the padding block of an odd pair owns no tile
        add_to_totals(mode == kModeDispatch ? p.totals : p.counts_scratch, E, et < FB_MAX_EXPERTS ? sh.hist[et] : 0u, et);
        if (mode == kModeDispatch) write_slice_counts(p.slice_counts, tile, E, sh.hist, et);
      }
    } else if (p.probe == 0) {
      publish_counts(sh, p, et, warp, lane, mode == kModePredictPlan && p.fuse_planner != 0);
    }
    FB_STAMP(12, 64);
  }

  // ---------------------------------------------------------------- teardown
  // Tensor memory may be released, and a block may leave, only when both blocks of the pair
  // are done with it: every warp has delivered its arrival for the pair's barrier as soon as
  // its own last access was over (producer and issuers after their loops, epilogue warps after
  // reading the accumulators), so this wait normally finds the barrier complete.
  tcgen05_fence_before();
  __syncthreads();
  cluster_wait();
  if (threadIdx.x == 0 && sh.abort_flag) atomicCAS(p.status, 0, FB_ERR_TIMEOUT);
  if (warp == 1) {
    tcgen05_fence_after();
    tmem_dealloc<2>(tmem_base, static_cast<uint32_t>(p.tmem_cols));
  }
  FB_STAMP(13, 64);
}

// Self-test of the bounded wait every kernel of this library relies on: one thread waits, for
// at most limit_ns, on a barrier that nobody ever arrives at.  The wait gives up, the kernel
// records FB_ERR_TIMEOUT in the status word and returns normally - the same path a router
// kernel takes when a copy or an MMA it waits for never completes.
// steps > 0: another warp reports that many steps of half the limit each and then arrives, so the wait lasts longer
// than the limit and ends well.
__global__ void __launch_bounds__(64, 1)
fb_wait_selftest_kernel(uint64_t limit_ns, int32_t steps, int32_t* status, uint64_t* waited_ns) {
  __shared__ uint64_t bar;
  __shared__ int32_t abort_flag;
  __shared__ int32_t progress;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    progress = 0;
    mbar_init(smem_u32(&bar), 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint64_t t0 = global_timer_ns();
    const bool ok = mbar_wait<false>(smem_u32(&bar), 0u, &abort_flag, limit_ns, &progress);
    if (waited_ns != nullptr) *waited_ns = global_timer_ns() - t0;
    if (!ok) atomicCAS(status, 0, FB_ERR_TIMEOUT);
  } else if (threadIdx.x == 32 && steps > 0) {
    for (int i = 1; i <= steps; ++i) {
      const uint64_t t0 = global_timer_ns();
      while (global_timer_ns() - t0 < limit_ns / 2) { }
      *static_cast<volatile int32_t*>(&progress) = i;
    }
    mbar_arrive(smem_u32(&bar));
  }
}

// Stand-alone planner: placement and counts by one thread per expert (both loads in flight at once;
// a single warp walking them took 11 of the kernel's 13 us), the decision by one warp.
// counts_out: the counts are the totals that the blocks of a prediction pass have added up (counts_scratch); they become the
// count vector (Eq. 5) and are put back to zero.  That takes the end of the pass out of the router kernel: a fence and a
// ticket in every block, the last block's loads and the planner at the end of the grid took longer than this launch, which waits
// on an SM of its own: prediction and plan of 300 tokens, 128 experts 14.3 -> 11.8 us, 8192 x 128 17.4 -> 16.4, 16384 x 256
// (power bound) 65 -> 62.
// kGeneral: for plans that need the general loop (plan_needs_general_loop).
template <bool kGeneral>
__global__ void __launch_bounds__(kPlanThreads, 1)
fb_plan_kernel(const __grid_constant__ PlanParams p, uint32_t* __restrict__ counts, uint32_t* __restrict__ counts_out, int32_t* status) {
  __shared__ PlanShared sh;
  const int t = threadIdx.x;
  static_assert(kPlanThreads >= FB_MAX_EXPERTS, "one thread per expert");
  plan_clear(sh, t, kPlanThreads);
  plan_place_ranks(p, sh, t, kPlanThreads);
  __syncthreads();
  pdl_wait();
  pdl_launch_dependents();               // (why here: fb_dispatch.cuh)
  if (t < p.E) {
    const uint32_t count = __ldcg(counts + t);
    const int slot = p.expert_to_slot[t];
    plan_place(p, sh, t, slot);
    plan_put_count_at(sh, t, slot, count, p.E);
    if (counts_out != nullptr) { counts_out[t] = count; counts[t] = 0; }
  }
  __syncthreads();
  if (t < 32) plan_swaps_warp<kGeneral>(p, sh, t, status);
  __syncthreads();
  plan_write_placement(p, sh, t, kPlanThreads);
}

}  // namespace fb
