// Dispatch index under the committed placement (stage 4 of the method): a stable
// counting sort of the T*k (token, expert) assignments by physical slot.  Positions
// come from prefix sums and population counts only - no atomic decides an output
// position - so the result is unique and reproducible.
//
// Input: the router kernel's top-k ids, its per-slice expert histogram
// slice_counts[slice][e] (slices_per_tile slices of slice_rows tokens per tile, one byte per expert: a
// token names an expert at most once, so a count is at most 128) and its totals per expert, which the router blocks add up in
// global memory.  One block per 128-token tile, or per run of consecutive tiles when there are more tiles than blocks.
// A block needs, besides the totals, the counts of the tiles before its own: it adds up the rows of the table before it or
// those from its first on, whichever are fewer.
//
// What bounds it: latency, not bandwidth (16 T k bytes of output are 2 MB at 16k tokens).  So
// everything a block needs from global memory is requested at once, before anything depends on it
// (placement, totals, first tile's ids, its part of the histogram table four experts per load), and the launch may
// overlap the end of the router kernel (programmatic dependent launch; layer calls back to back without and with it: 512
// tokens, 8 experts 12.4 and 9.7 us, 1000 x 128 16.5 and 14.1, 8192 x 128 22.7 and 20.3, 131072 x 128 no difference).
// The next kernel of the stream may set itself up, and a router kernel bring rows into L2 (prefetch_operands), while a
// kernel of this file or the planner kernel runs - but not before its wait is over: allowed earlier, a whole chain of small kernels
// starts during the main loop of the router kernel before them, and the next router kernel takes SMs and bandwidth
// from it (layer calls back to back, allowed before and after the wait: 1733 tokens, 256 experts 31.6 and 30.7 us, 1000 x 128
// 19.8 and 18.9; a shard's six launches 58.0 and 56.6).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/freebalance.h"
#include "fb_planner.cuh"
#include "fb_ptx.cuh"

// Phase time stamps (builds with -DFB_TIMING only; see fb_set_stamp_buffer): one designated
// thread per role writes %globaltimer (slot i) and clock64 (slot 32 + i) of its block at the
// phase boundaries below.  Without the flag the macro is empty and the kernels carry none of it.
//   0 block start          1 set-up done            2 accumulators complete  3 keys computed
//   4 barrier              5 groups chosen          7 candidates collected   8 candidates ranked
//   9 top-k read back     10 outputs written       11 counts published      12 planner done
//  13 block exit          14 first load issued     15 last load issued      16 first operands landed
//  17 last MMA issued     18 planner entered       19 rank loads formed    20 greedy loop left
// and in the dispatch-index kernel
//  21 block start         22 wait over             23 tables read           24 barrier
//  25 totals formed       26 planner done          27 offsets formed        28 block exit
#ifdef FB_TIMING
#define FB_STAMP(i, who)                                                                    \
  do {                                                                                      \
    if (p.stamps != nullptr && threadIdx.x == (who)) {                                      \
      unsigned long long* st_ = p.stamps + static_cast<size_t>(blockIdx.x) * 64;           \
      st_[i] = global_timer_ns();                                                           \
      st_[32 + (i)] = static_cast<unsigned long long>(clock64());                           \
    }                                                                                       \
  } while (0)
#else
#define FB_STAMP(i, who) do { } while (0)
#endif

namespace fb {

constexpr int kDispatchThreads = 1024;
constexpr int kDispatchTile = 128;       // must equal the router kernel's tile height
constexpr int kDispatchWarps = kDispatchThreads / 32;
// Rows of a tile that one of `pieces` blocks finishes: even (rows are selected two at a time), the last block has
// the rest.
__host__ __device__ constexpr int slice_rows(int pieces) { return (kDispatchTile + 2 * pieces - 1) / (2 * pieces) * 2; }
constexpr int kDispatchBatch = 4;        // tiles a block works on at a time
static_assert(kDispatchTile * FB_MAX_TOPK == kDispatchThreads, "one thread per assignment of a tile");
// Bytes of one row of the histogram table: 16-byte units (a lane reads four experts at once, see add_rows).
__host__ __device__ constexpr int slice_row_bytes(int E) { return (E + 15) & ~15; }

struct DispatchParams {
  int32_t T, k, E, R, num_tiles;
  int32_t num_slices, slices_per_tile;
  int32_t per_rank;                // E / R
  const int32_t* topk_ids;         // [T][k]
  const uint8_t* slice_counts;     // [num_slices][slice_row_bytes(E)]
  // [FB_MAX_EXPERTS] of the normal pass, then (fb_dispatch_kernel<true> only) as many of the early pass; what the grid has
  // read its last block puts back to zero
  uint32_t* totals;
  uint32_t* ticket;                // zero on entry, zero again on exit
  const int32_t* expert_to_slot;   // [E]
  uint32_t* slot_offsets;          // [E+1]
  uint32_t* rank_offsets;          // [R+1]
  int32_t* perm;                   // [T*k]
  int32_t* inv_perm;               // [T*k]
  uint32_t* rank_load;             // [R]
  int32_t* status;
  // fb_dispatch_kernel<true>: the count vector and the plan that are formed from the early pass's totals, and whose
  // output placement the index is made under
  uint32_t* counts_out;            // [E]
  PlanParams plan;
  unsigned long long* stamps;      // [blocks][64] phase time stamps (FB_TIMING builds) or nullptr
};

// Four bytes as two pairs of 16-bit counters.
__device__ __forceinline__ void add_bytes(uint32_t& even, uint32_t& odd, uint32_t w) {
  even += w & 0x00ff00ffu;
  odd += (w >> 8) & 0x00ff00ffu;
}

// Column sums over rows [first, last) of the histogram table.  A row is W = row_bytes / 4 words of four experts; a
// warp reads 32 / W rows at a time (one where W > 16), lane l word l % W - and word l + 32 where W > 32 - and the warps take
// turns, so that a lane adds one or two words per step and no sums have to be exchanged but those of the rows of one
// step.  (With 16 bytes per lane, eight rows per warp and step, the sums went through 32 shuffles per warp.)
struct RowSums {
  uint32_t even[2], odd[2];          // two 16-bit counters each: bytes 0 and 2, bytes 1 and 3 of the lane's words
};
__device__ __forceinline__ RowSums add_rows(const uint8_t* table, int row_bytes, int first, int last, int warp, int warps,
                                            int lane) {
  RowSums s = {{0, 0}, {0, 0}};
  const int W = row_bytes >> 2, at_once = W <= 16 ? 32 / W : 1;
  const int sub = W <= 16 ? lane / W : 0, word = W <= 16 ? lane % W : lane;
  const bool one = sub < at_once && word < W, two = lane + 32 < W;
  const uint8_t* at = table + static_cast<size_t>(word) * 4;
#pragma unroll 4
  for (int r = first + warp * at_once + sub; r < last; r += warps * at_once) {
    const uint8_t* row = at + static_cast<size_t>(r) * row_bytes;
    const uint32_t v = one ? __ldcg(reinterpret_cast<const uint32_t*>(row)) : 0u;
    const uint32_t w = two ? __ldcg(reinterpret_cast<const uint32_t*>(row + 128)) : 0u;
    add_bytes(s.even[0], s.odd[0], v);
    add_bytes(s.even[1], s.odd[1], w);
  }
  __syncwarp();
  if (W <= 16) {                     // the rows of one step: lanes W apart
    for (int off = at_once / 2 * W; off >= W; off = off / W / 2 * W) {
      s.even[0] += __shfl_down_sync(0xffffffffu, s.even[0], off);
      s.odd[0] += __shfl_down_sync(0xffffffffu, s.odd[0], off);
    }
  }
  return s;
}
// ... to part[word] = experts 4 w, 4 w + 2 in word 2 w and the two others in word 2 w + 1.
__device__ __forceinline__ void store_row_sums(const RowSums& s, uint32_t* part, int row_bytes, int lane) {
  const int W = row_bytes >> 2;
  if (lane < W) *reinterpret_cast<uint2*>(part + 2 * lane) = make_uint2(s.even[0], s.odd[0]);
  if (lane + 32 < W) *reinterpret_cast<uint2*>(part + 2 * lane + 64) = make_uint2(s.even[1], s.odd[1]);
}

template <bool kFirst, class A, class B> struct Choose { using type = A; };
template <class A, class B> struct Choose<false, A, B> { using type = B; };

// Rows of a tile below `row` among those marked in m (128 bits).
__device__ __forceinline__ uint32_t rows_before(const uint4& m, int row) {
  const int w = row >> 5;
  const uint32_t low = (1u << (row & 31)) - 1u;
  return __popc(m.x & (w > 0 ? 0xffffffffu : low)) + __popc(m.y & (w > 1 ? 0xffffffffu : (w == 1 ? low : 0u))) +
         __popc(m.z & (w > 2 ? 0xffffffffu : (w == 2 ? low : 0u))) + __popc(m.w & (w == 3 ? low : 0u));
}

// Exclusive prefix of `count` over the slots, thread t for slot t (0 beyond the last); the whole block calls
// it.  Returns the prefix; *all receives the total in thread E - 1.  warp_sum: 8 words that nobody else uses
// until the next barrier.  (By one warp with 8 slots per lane it took 1 us.)
__device__ __forceinline__ uint32_t block_prefix(uint32_t count, uint32_t* warp_sum, int t, uint32_t* all) {
  const int warp = t >> 5, lane = t & 31;
  uint32_t incl = count;
  if (warp < FB_MAX_EXPERTS / 32) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += o;
    }
    if (lane == 31) warp_sum[warp] = incl;
  }
  __syncthreads();
  if (warp < FB_MAX_EXPERTS / 32) {
#pragma unroll
    for (int w = 0; w < FB_MAX_EXPERTS / 32; ++w) incl += w < warp ? warp_sum[w] : 0u;
  }
  *all = incl;
  return incl - count;
}

__device__ __forceinline__ void write_offsets(const DispatchParams& p, const uint32_t* offs, int t) {
  // (with loops over E and R and a division by R in block 0: layer call 1733 x 256 27.8 -> 27.1 us, 1000 x 128 14.9 -> 14.5,
  // 40 x 128 13.4 -> 12.9)
  static_assert(kDispatchThreads > FB_MAX_EXPERTS + FB_MAX_RANKS + 1, "one element per thread");
  const int m = p.per_rank, r = t - (kDispatchThreads - FB_MAX_RANKS - 1);      // ranks: the last threads
  if (t <= p.E) p.slot_offsets[t] = offs[t];
  if (r >= 0 && r <= p.R) {
    p.rank_offsets[r] = offs[r * m];
    if (r < p.R) p.rank_load[r] = offs[(r + 1) * m] - offs[r * m];
  }
}

// The totals have been read by all blocks: the last one puts them back to zero for the next call (kBoth: those of both
// passes; otherwise the early pass's words are another call's).  By one warp, after a barrier behind the block's reads
// (their values have arrived: nothing of this grid is still to be read).
__device__ __forceinline__ uint32_t take_index_ticket(const DispatchParams& p, int lane) {
  return lane == 0 ? atomicAdd(p.ticket, 1u) : 0u;
}
template <bool kBoth>
__device__ __forceinline__ void clear_totals(const DispatchParams& p, uint32_t ticket, int lane) {
  if (__shfl_sync(0xffffffffu, ticket, 0) != gridDim.x - 1) return;
  for (int i = lane; i < (kBoth ? 2 : 1) * FB_MAX_EXPERTS; i += 32) p.totals[i] = 0;
  if (lane == 0) *p.ticket = 0;
}

// One tile per block (at most as many tiles as SMs).  The work per expert does not depend on the
// placement; the slots come in with one scan at the end.
// kPlan: the swap planner runs in here as well, in every block (its decisions are integer and reproducible,
// so no block waits for another; block 0 writes counts and plan, block 1 - or block 0 alone - the placement).  Used where a
// layer launch runs both passes at the same time: electing the last block of the early pass and planning in
// it were 3 to 5 us at the end of the router kernel with every other SM idle.
// The first warp plans as soon as totals and placement have arrived; the others add up the table and find every
// assignment's place among its tile's meanwhile.  Against totals out of the tables of both passes, with the planner behind
// them: 8192 x 128 24.2 -> 23.0 us, 1733 x 256 29.1 -> 28.1, 1000 x 128 17.6 -> 16.7, 40 x 128 15.1 -> 14.7.
constexpr uint32_t kIndexPlanBarrier = 1, kIndexTableBarrier = 2;     // named barriers
template <bool kPlan>
__global__ void __launch_bounds__(kDispatchThreads, 1)
fb_dispatch_kernel(const __grid_constant__ DispatchParams p) {
  struct Empty {};
  __shared__ int32_t expert_at[FB_MAX_EXPERTS];    // slot -> expert
  __shared__ uint32_t base[FB_MAX_EXPERTS];        // expert: assignments in earlier tiles; then the tile's first position
  __shared__ uint32_t total[FB_MAX_EXPERTS];       // expert: assignments in all tiles
  __shared__ uint32_t offs[FB_MAX_EXPERTS + 1];    // exclusive prefix of total over slots
  __shared__ uint4 mask[FB_MAX_EXPERTS];           // rows of the tile that chose the expert
  __shared__ uint32_t warp_sum[FB_MAX_EXPERTS / 32];
  __shared__ alignas(8) uint32_t part[kDispatchWarps][FB_MAX_EXPERTS / 2];    // see store_row_sums
  __shared__ typename Choose<kPlan, PlanShared, Empty>::type plan;
  __shared__ int32_t bad;

  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int E = p.E, k = p.k;
  const int tile = static_cast<int>(blockIdx.x);
  FB_STAMP(21, 0);
  if (t == 0) bad = 0;
  if (t < FB_MAX_EXPERTS) { expert_at[t] = -1; mask[t] = make_uint4(0, 0, 0, 0); }
  if constexpr (kPlan) {
    plan_clear(plan, t, kDispatchThreads);
    plan_place_ranks(p.plan, plan, t, kDispatchThreads);
  }
  // Thread t owns assignment t of the tile: row t / k, choice t % k (exact for t < 8192, k <= 8).
  const int row = (t * ((65536 + k - 1) / k)) >> 16;
  const long long flat = static_cast<long long>(tile) * kDispatchTile * k + t;
  const long long n_assign = static_cast<long long>(p.T) * k;
  const bool owns = t < kDispatchTile * k && flat < n_assign;
  const int row_bytes = slice_row_bytes(E), W = row_bytes >> 2;
  const int first_slice = tile * p.slices_per_tile;
  const bool later = 2 * first_slice > p.num_slices;               // fewer rows from this tile's first on than before it
  const int row_first = later ? first_slice : 0, row_last = later ? p.num_slices : first_slice;
  __syncthreads();
  pdl_wait();                                    // from here on: what the router kernel wrote
  pdl_launch_dependents();
  FB_STAMP(22, 0);
  // ---- everything the block needs from global memory, before anything depends on it
  const int my_slot = t < E ? p.expert_to_slot[t] : 0;
  const uint32_t my_total = t < E ? __ldcg(p.totals + t) : 0u;
  const uint32_t my_early = kPlan && t < E ? __ldcg(p.totals + FB_MAX_EXPERTS + t) : 0u;
  int e = owns ? p.topk_ids[flat] : 0;
#ifdef FB_DEBUG
  if (e < 0 || e >= E) atomicCAS(p.status, 0, FB_ERR_INTERNAL);         // an expert id outside [0, E)
#endif
  if (e < 0 || e >= E) e = 0;
  if (t < E) {
    total[t] = my_total;
    if constexpr (kPlan) {
      plan_place(p.plan, plan, t, my_slot);
      plan_put_count_at(plan, t, my_slot, my_early, E);
      if (tile == 0) p.counts_out[t] = my_early;
    } else {
      if (my_slot < 0 || my_slot >= E || atomicExch(&expert_at[my_slot], t) != -1) bad = 1;
    }
  }
  if (owns) atomicOr(reinterpret_cast<uint32_t*>(&mask[e]) + (row >> 5), 1u << (row & 31));
  if constexpr (kPlan) {
    if (warp < FB_MAX_EXPERTS / 32) named_bar_sync(kIndexPlanBarrier, FB_MAX_EXPERTS);
    FB_STAMP(25, 0);
    if (warp == 0) {
      named_bar_arrive(kIndexTableBarrier, kDispatchThreads);
      plan_swaps_warp<false>(p.plan, plan, lane, p.status, tile == 0);
    }
  }
  uint32_t ticket = 0, ahead = 0;
  if (!kPlan || warp != 0) {
    constexpr int kFirst = kPlan ? 1 : 0;          // the first warp that adds rows
    store_row_sums(add_rows(p.slice_counts, row_bytes, row_first, row_last, warp - kFirst, kDispatchWarps - kFirst, lane),
                   part[warp], row_bytes, lane);
    FB_STAMP(23, 32);
    named_bar_sync(kIndexTableBarrier, kDispatchThreads);
    FB_STAMP(24, 32);
    if (warp == kDispatchWarps - 1) ticket = take_index_ticket(p, lane);
    const int j = t - 32 * kFirst;
    if (j < 2 * W) {
      uint32_t s0 = 0, s1 = 0;
#pragma unroll 8
      for (int w = kFirst; w < kDispatchWarps; ++w) {
        const uint32_t v = part[w][j];
        s0 += v & 0xffffu; s1 += v >> 16;
      }
      const int e0 = 4 * (j >> 1) + (j & 1), e1 = e0 + 2;
      if (e0 < E) base[e0] = later ? total[e0] - s0 : s0;
      if (e1 < E) base[e1] = later ? total[e1] - s1 : s1;
    }
    ahead = rows_before(mask[e], row);
  }
  __syncthreads();
  FB_STAMP(26, 0);
  if (kPlan && warp == 0) ahead = rows_before(mask[e], row);
  bool usable = bad == 0;
  if constexpr (kPlan) usable = plan.bad == 0;
  uint32_t count = 0, all = 0;
  int expert = 0;
  if (t < E && usable) {
    if constexpr (kPlan) expert = plan.bad_range ? plan.expert_at[t] : static_cast<int>(plan.slot_cnt[t] & 0xffu);
    else expert = expert_at[t];
    count = total[expert];
  }
  const uint32_t first = block_prefix(count, warp_sum, t, &all);
  if (t < E && usable) {
    offs[t] = first;
    base[expert] += first;
    if (t == E - 1) offs[E] = all;
  }
  __syncthreads();
  FB_STAMP(27, 0);
  if constexpr (kPlan)                             // (not by the block that writes the offsets, where there is another)
    if (tile == (gridDim.x > 1 ? 1 : 0)) plan_write_placement(p.plan, plan, t, kDispatchThreads);
  if (usable) {
    if (tile == 0) write_offsets(p, offs, t);
    if (owns) {
      const long long pos = static_cast<long long>(base[e]) + ahead;
#ifdef FB_DEBUG
      if (pos < 0 || pos >= n_assign) atomicCAS(p.status, 0, FB_ERR_INTERNAL);   // a position outside [0, T k)
#endif
      if (pos < n_assign) {
        p.perm[pos] = static_cast<int32_t>(flat);
        p.inv_perm[flat] = static_cast<int32_t>(pos);
      }
    }
  } else if (!kPlan && t == 0 && tile == 0) {      // not a bijection: report (the planner has), write no index
    atomicCAS(p.status, 0, FB_ERR_BAD_PLACEMENT);
  }
  if (warp == kDispatchWarps - 1) clear_totals<kPlan>(p, ticket, lane);
  FB_STAMP(28, 0);
}

// A run of consecutive tiles per block (more tiles than SMs).
__global__ void __launch_bounds__(kDispatchThreads, 1)
fb_dispatch_runs_kernel(const __grid_constant__ DispatchParams p) {
  constexpr int kBatch = kDispatchBatch;
  __shared__ int32_t slot_of[FB_MAX_EXPERTS];
  __shared__ int32_t owner[FB_MAX_EXPERTS];
  __shared__ uint32_t gbase[FB_MAX_EXPERTS];       // position of the slot's first assignment of this batch of tiles
  __shared__ uint32_t total[FB_MAX_EXPERTS];       // assignments to this slot in all tiles
  __shared__ uint32_t warp_sum[FB_MAX_EXPERTS / 32];
  __shared__ uint32_t offs[FB_MAX_EXPERTS + 1];    // exclusive prefix of total over slots; later: of the batch's counts
  __shared__ uint16_t ahead_of[kBatch][FB_MAX_EXPERTS];   // the batch's assignments to this slot in earlier tiles
  // The per-warp sums of the histogram table are read before the tile loop starts and share their
  // memory with what the loop works on.
  __shared__ alignas(16) union {
    uint32_t part[kDispatchWarps][FB_MAX_EXPERTS / 2];      // see store_row_sums
    struct {
      uint4 mask[kBatch][FB_MAX_EXPERTS];                   // rows of the tile that go to the slot
      uint32_t sorted[kBatch * kDispatchThreads];   // the batch's assignments in slot order: slot << 16 | tile, thread
    } b;
  } u;
  __shared__ int32_t bad;

  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int E = p.E, k = p.k;
  // This block's tiles: a contiguous range, so that "assignments in earlier tiles" can be carried
  // from one tile to the next instead of being summed again.
  const int per_block = (p.num_tiles + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);
  const int tile_begin = static_cast<int>(blockIdx.x) * per_block;
  const int tile_end = min(p.num_tiles, tile_begin + per_block);
  if (t == 0) bad = 0;
  if (t < FB_MAX_EXPERTS) owner[t] = -1;
  // Thread t owns assignment t of the tile: row t / k, choice t % k (exact for t < 8192, k <= 8).
  const int row = (t * ((65536 + k - 1) / k)) >> 16;
  const long long n_assign = static_cast<long long>(p.T) * k;
  auto load_id = [&](int tile) -> int {
    const long long flat = static_cast<long long>(tile) * kDispatchTile * k + t;
    if (tile >= tile_end || t >= kDispatchTile * k || flat >= n_assign) return -1;
    const int e = p.topk_ids[flat];
#ifdef FB_DEBUG
    if (e < 0 || e >= E) atomicCAS(p.status, 0, FB_ERR_INTERNAL);       // an expert id outside [0, E)
#endif
    return (e < 0 || e >= E) ? 0 : e;
  };
  pdl_wait();                                    // from here on: what the router kernel wrote
  pdl_launch_dependents();
  const int my_slot_in = t < E ? p.expert_to_slot[t] : 0;
  int ids[kBatch];
#pragma unroll
  for (int i = 0; i < kBatch; ++i) ids[i] = load_id(tile_begin + i);
  const uint32_t my_total = t < E ? __ldcg(p.totals + t) : 0u;
  // ---- column sums of the histogram table before this block's first slice, or from it on.  16-bit counters: a lane
  // adds 500 slices of at most 128 at most between two flushes.
  const int row_bytes = slice_row_bytes(E), W = row_bytes >> 2;
  const int first_slice = min(tile_begin * p.slices_per_tile, p.num_slices);
  const bool later = 2 * first_slice > p.num_slices;
  const int row_first = later ? first_slice : 0, row_last = later ? p.num_slices : first_slice;
  constexpr int kFlush = 500 * kDispatchWarps;
  uint32_t sum0 = 0, sum1 = 0;                   // thread j < 2 W: experts 4 (j / 2) + j % 2 and that + 2
  for (int s_base = row_first; s_base < row_last; s_base += kFlush) {
    const RowSums sums = add_rows(p.slice_counts, row_bytes, s_base, min(row_last, s_base + kFlush), warp, kDispatchWarps, lane);
    if (s_base > row_first) __syncthreads();     // the previous flush has been read
    store_row_sums(sums, u.part[warp], row_bytes, lane);
    __syncthreads();
    if (t < 2 * W) {
#pragma unroll 8
      for (int w = 0; w < kDispatchWarps; ++w) {
        const uint32_t v = u.part[w][t];
        sum0 += v & 0xffffu; sum1 += v >> 16;
      }
    }
  }
  if (t < E) {
    if (my_slot_in < 0 || my_slot_in >= E) bad = 1;
    else if (atomicExch(&owner[my_slot_in], t) != -1) bad = 1;
    slot_of[t] = (my_slot_in < 0 || my_slot_in >= E) ? 0 : my_slot_in;
    total[slot_of[t]] = my_total;
  }
  __syncthreads();
  const uint32_t ticket = warp == kDispatchWarps - 1 ? take_index_ticket(p, lane) : 0u;
  if (bad || tile_begin >= tile_end) {
    if (warp == kDispatchWarps - 1) clear_totals<false>(p, ticket, lane);
    if (bad && t == 0 && blockIdx.x == 0) atomicCAS(p.status, 0, FB_ERR_BAD_PLACEMENT);   // not a bijection: report, write nothing
    return;
  }
  if (t < 2 * W) {
    const int e0 = 4 * (t >> 1) + (t & 1), e1 = e0 + 2;
    if (e0 < E) { const int sl = slot_of[e0]; gbase[sl] = later ? total[sl] - sum0 : sum0; }
    if (e1 < E) { const int sl = slot_of[e1]; gbase[sl] = later ? total[sl] - sum1 : sum1; }
  }
  static_assert(kDispatchThreads == kDispatchBatch * FB_MAX_EXPERTS, "one mask per thread");
  u.b.mask[t / FB_MAX_EXPERTS][t % FB_MAX_EXPERTS] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  auto mark_rows = [&]() {
#pragma unroll
    for (int i = 0; i < kBatch; ++i)
      if (ids[i] >= 0) {
        uint32_t* m = reinterpret_cast<uint32_t*>(&u.b.mask[i][slot_of[ids[i]]]);
        atomicOr(m + (row >> 5), 1u << (row & 31));
      }
  };
  mark_rows();
  uint32_t all = 0;
  const uint32_t first = block_prefix(t < E ? total[t] : 0u, warp_sum, t, &all);
  if (t < E) {
    offs[t] = first;
    gbase[t] += first;
    if (t == E - 1) offs[E] = all;
  }
  if (blockIdx.x == 0) {
    __syncthreads();
    write_offsets(p, offs, t);
  }
  // Up to four tiles at a time.  With more than one, their assignments are first put into slot
  // order in shared memory, so that perm is written in runs (4-byte stores to as many sectors as
  // threads took 4 us of the 18 us at 131072 tokens); a single tile has runs of a few entries only and writes directly.
  for (int tile0 = tile_begin; tile0 < tile_end; tile0 += kBatch) {
    const bool several = tile_end - tile0 > 1;                  // (the same for the whole block)
    __syncthreads();                                            // the masks are complete, the offsets written
    uint32_t run = 0;
    if (several) {
      if (t < E) {
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
          ahead_of[i][t] = static_cast<uint16_t>(run);
          const uint4 m = u.b.mask[i][t];
          run += __popc(m.x) + __popc(m.y) + __popc(m.z) + __popc(m.w);
        }
      }
      const uint32_t at = block_prefix(run, warp_sum, t, &all);
      if (t < E) {
        offs[t] = at;
        if (t == E - 1) offs[E] = all;
      }
      __syncthreads();
    }
    int next_ids[kBatch];
#pragma unroll
    for (int i = 0; i < kBatch; ++i) next_ids[i] = load_id(tile0 + kBatch + i);
#pragma unroll
    for (int i = 0; i < kBatch; ++i) {
      if (ids[i] < 0) continue;
      const int my_slot = slot_of[ids[i]];
      uint32_t ahead = rows_before(u.b.mask[i][my_slot], row);
      if (several) ahead += ahead_of[i][my_slot];
      const long long pos = static_cast<long long>(gbase[my_slot]) + ahead;
      const long long flat = static_cast<long long>(tile0 + i) * kDispatchTile * k + t;
#ifdef FB_DEBUG
      if (pos < 0 || pos >= n_assign || flat >= n_assign || my_slot < 0 || my_slot >= E)
        atomicCAS(p.status, 0, FB_ERR_INTERNAL);                          // a position outside [0, T k) or a slot outside [0, E)
#endif
      if (pos < n_assign) {
        p.inv_perm[flat] = static_cast<int32_t>(pos);
        if (!several) p.perm[pos] = static_cast<int32_t>(flat);
      }
      if (several) {
        const uint32_t at = offs[my_slot] + ahead;
        if (at < kBatch * kDispatchThreads)
          u.b.sorted[at] = static_cast<uint32_t>(my_slot) << 16 | static_cast<uint32_t>(i) << 10 | static_cast<uint32_t>(t);
      }
    }
    if (!several) break;
    __syncthreads();
    const uint32_t count = min(offs[E], static_cast<uint32_t>(kBatch * kDispatchThreads));
    for (uint32_t at = t; at < count; at += kDispatchThreads) {
      const uint32_t v = u.b.sorted[at];
      const uint32_t slot = v >> 16;
      const long long pos = static_cast<long long>(gbase[slot]) + (at - offs[slot]);
      if (pos < n_assign)
        p.perm[pos] = static_cast<int32_t>((tile0 + static_cast<int>((v >> 10) & 3u)) * kDispatchTile * k + static_cast<int>(v & 1023u));
    }
    if (tile0 + kBatch >= tile_end) break;
    u.b.mask[t / FB_MAX_EXPERTS][t % FB_MAX_EXPERTS] = make_uint4(0, 0, 0, 0);
    __syncthreads();
    if (t < E) gbase[t] += run;
#pragma unroll
    for (int i = 0; i < kBatch; ++i) ids[i] = next_ids[i];
    mark_rows();
    __syncthreads();
  }
  if (warp == kDispatchWarps - 1) clear_totals<false>(p, ticket, lane);
}

// ---- token-sharded dispatch (several GPUs, each with a contiguous token range in rank order)
// A shard's dispatch index is local.  The order of the whole batch is by (slot, token), so in
// slot p the assignments of earlier ranks come first: the whole-batch position of a local
// assignment at local position q in slot p is
//     G[p] + sum_{r' < rank} counts[r'][p] + (q - local_offsets[p]),
// G = exclusive prefix over slots of the counts summed over all ranks.  counts[r][p] is what the
// ranks exchange (an all-gather of E words per rank).

// Both kernels are a few microseconds of latency: they start under the end of the kernel before them.

// counts[p] = number of local assignments in slot p
__global__ void fb_slot_counts_kernel(const uint32_t* __restrict__ slot_offsets, int E, uint32_t* __restrict__ counts) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_wait();
  pdl_launch_dependents();
  if (p < E) counts[p] = __ldcg(slot_offsets + p + 1) - __ldcg(slot_offsets + p);
}

constexpr int kGlobalizeThreads = 256;   // >= FB_MAX_EXPERTS: one thread per slot for the shifts

struct GlobalizeParams {
  int32_t T, k, E, R, world, rank;
  int32_t per_rank;                  // E / R
  const uint32_t* counts_all;        // [world][E]
  const uint32_t* local_offsets;     // [E+1]
  const int32_t* topk_ids;           // [T][k] (local)
  const int32_t* expert_to_slot;     // [E]
  int32_t* inv_perm;                 // [T*k] in: local positions, out: whole-batch positions
  uint32_t* slot_offsets;            // [E+1] out (whole batch)
  uint32_t* rank_offsets;            // [R+1] out
  uint32_t* rank_load;               // [R]   out
};

// Exclusive prefix by warp scans and all loads up front: with one thread adding 256 slots in turn and
// the assignments loaded behind it the kernel took 9.6 us, now 3.9 (2048 tokens, 256 slots, 8 ranks).
__global__ void __launch_bounds__(kGlobalizeThreads)
fb_dispatch_globalize_kernel(const __grid_constant__ GlobalizeParams p) {
  __shared__ uint32_t shift[FB_MAX_EXPERTS];
  __shared__ uint32_t G[FB_MAX_EXPERTS + 1];
  __shared__ uint32_t warp_sum[kGlobalizeThreads / 32];
  __shared__ int32_t slot_of[FB_MAX_EXPERTS];
  static_assert(kGlobalizeThreads == FB_MAX_EXPERTS, "one thread per slot");
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  pdl_wait();
  pdl_launch_dependents();
  const long long n = static_cast<long long>(p.T) * p.k;
  long long q = static_cast<long long>(blockIdx.x) * kGlobalizeThreads + t;
  int e = q < n ? p.topk_ids[q] : -1;
  uint32_t pos = q < n ? static_cast<uint32_t>(p.inv_perm[q]) : 0u;
  const int my_slot = t < p.E ? p.expert_to_slot[t] : -1;
  const uint32_t local = t < p.E ? p.local_offsets[t] : 0u;
  uint32_t before = 0, total = 0;
  if (t < p.E) {
#pragma unroll 8
    for (int r = 0; r < p.world; ++r) {
      const uint32_t c = p.counts_all[static_cast<size_t>(r) * p.E + t];
      before += r < p.rank ? c : 0u;
      total += c;
    }
  }
  uint32_t incl = total;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += o;
  }
  if (lane == 31) warp_sum[warp] = incl;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < kGlobalizeThreads / 32; ++w) incl += w < warp ? warp_sum[w] : 0u;
  if (t < p.E) {
    G[t] = incl - total;
    if (t == p.E - 1) G[p.E] = incl;
    shift[t] = incl - total + before - local;
    slot_of[t] = my_slot;
  }
  __syncthreads();
  if (blockIdx.x == 0) {
    const int m = p.per_rank;
    for (int s = t; s <= p.E; s += kGlobalizeThreads) p.slot_offsets[s] = G[s];
    for (int r = t; r <= p.R; r += kGlobalizeThreads) p.rank_offsets[r] = G[r * m];
    for (int r = t; r < p.R; r += kGlobalizeThreads) p.rank_load[r] = G[(r + 1) * m] - G[r * m];
  }
  while (q < n) {
    const int s = (e >= 0 && e < p.E) ? slot_of[e] : -1;
    if (s >= 0 && s < p.E) p.inv_perm[q] = static_cast<int32_t>(pos + shift[s]);
    q += static_cast<long long>(gridDim.x) * kGlobalizeThreads;
    if (q < n) { e = p.topk_ids[q]; pos = static_cast<uint32_t>(p.inv_perm[q]); }
  }
}

}  // namespace fb
