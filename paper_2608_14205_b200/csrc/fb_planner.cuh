// Budgeted greedy expert-swap planner (Algorithm 1 lines 2-8, Eqs. 6-9), decided by one
// warp: of the planner kernel (alone or behind a prediction pass), of every block of the dispatch-index kernel
// (layer calls with one tile per SM), or, with more tiles than the GPU holds at once, of the persistent router kernel's last
// pair (a warp that is idle there) or of the other router kernels' last block.  Integer arithmetic only, so
// every block and every rank that replays it on the same count vector gets the same plan.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/freebalance.h"
#include "fb_ptx.cuh"

namespace fb {

constexpr int kPlanThreads = 256;         // the stand-alone planner kernel: one thread per expert; one warp decides
constexpr uint32_t kPlanBarrierId = 1;    // named barrier of the router kernel's epilogue warps

struct PlanParams {
  int32_t E, R;
  int32_t per_rank;                     // E / R, and what replaces the division by it (rank_of_slot); host
  uint32_t per_rank_inv;
  uint32_t max_swaps;
  uint64_t global_ns, rank_ns, link_ns;
  uint32_t tau_tokens;
  uint32_t gamma_num, gamma_den;
  uint64_t alpha_ns[2];
  uint64_t fs_per_byte[2];
  uint64_t uniform_cost_ns[2];          // Eq. 9 evaluated on the host for the uniform expert size
  uint64_t uniform_link_cap[2];         // link_ns / uniform_cost_ns: swaps one link can carry (host)
  uint32_t swap_cap;                    // max_swaps, or fewer if the global budget carries fewer (one cost class only; host)
  int32_t books;                        // the uniform loop has to keep books: two cost classes, or a per-rank or
                                        // per-link budget that can stop a swap the global one admits (host)
  int32_t ranks_per_node;
  int32_t mode;                         // fb_plan_mode
  int32_t frontier_width;               // FB_PLAN_WIDE: ranks taken from each end of the load order (1..4)
  const uint64_t* expert_bytes_table;   // device [E] or nullptr
  const int32_t* expert_to_slot;        // device [E]
  int32_t* expert_to_slot_out;          // device [E]
  fb_swap* swaps;                       // device [max_swaps]
  int32_t* n_swaps;                     // device [1]
  uint32_t* load_before;                // device [R]
  uint32_t* load_after;                 // device [R]
};

// s / per_rank for a slot s < 256: with inv = ceil(65536 / m) the quotient is at most s / 65536 < 1 / 256 too large, and
// the fraction of s / m is at most 1 - 1 / m.
__host__ __device__ constexpr uint32_t per_rank_inverse(int m) { return (65536u + static_cast<uint32_t>(m) - 1u) / static_cast<uint32_t>(m); }
__device__ __forceinline__ int rank_of_slot(const PlanParams& p, int s) {
  return static_cast<int>(static_cast<uint32_t>(s) * p.per_rank_inv >> 16);
}

// Phase stamps of the planner (FB_TIMING builds only): 18 planner entered, 19 rank loads formed,
// 20 greedy loop left.
#ifdef FB_TIMING
#define FB_PLAN_STAMP(i)                                                                    \
  do {                                                                                      \
    if (stamps != nullptr && lane == 0) {                                                   \
      unsigned long long t_;                                                                \
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_));                                \
      stamps[i] = t_;                                                                       \
      stamps[32 + (i)] = static_cast<unsigned long long>(clock64());                        \
    }                                                                                       \
  } while (0)
#else
#define FB_PLAN_STAMP(i) do { } while (0)
#endif

struct PlanCandidate {
  long long benefit;                    // gamma_den * (Phi(L) - Phi(L')), > 0 when valid
  unsigned long long cost;              // C(s) in ns, >= 1
  int32_t a, b;                         // source and destination rank
  int32_t ea, eb;                       // ea < 0: no candidate
};

constexpr int kMaxFrontierWidth = 4;

struct PlanShared {
  uint32_t cnt[FB_MAX_EXPERTS];
  int32_t slot_of[FB_MAX_EXPERTS];       // expert -> slot (current placement)
  int32_t expert_at[FB_MAX_EXPERTS];     // slot -> expert
  uint8_t moved[FB_MAX_EXPERTS];
  // fast loop: one word per slot - the expert placed there in bits 0..7, twice its count above (kSlotMoved in the
  // place of a count once the expert has moved)
  alignas(16) uint32_t slot_cnt[FB_MAX_EXPERTS];
  uint8_t rank_of[FB_MAX_EXPERTS];       // expert -> rank under the placement as given
  uint8_t node_of[FB_MAX_RANKS];         // rank -> node (all 0 when every rank is in one node)
  uint32_t load[FB_MAX_RANKS];           // rank loads under the placement as given
  unsigned long long rank_spent[FB_MAX_RANKS];
  uint32_t link_key[FB_MAX_EXPERTS / 2]; // one entry per accepted swap
  unsigned long long link_cost[FB_MAX_EXPERTS / 2];
  int32_t bad;                           // the placement is not a bijection
  int32_t bad_range;                     // a count beyond the planner's range
  int32_t fast;                          // the fast loop ran: the placement is in slot_cnt, not in expert_at
};

constexpr uint32_t kSlotMoved = 1u << 22;       // as a count
static_assert(2 * FB_MAX_COUNT_SUM <= kSlotMoved && FB_MAX_EXPERTS <= 256, "slot word layout");
__device__ __forceinline__ uint32_t slot_word(uint32_t count, int expert) { return count << 9 | static_cast<uint32_t>(expert); }

// true if x is a better choice than y: larger benefit / cost, compared exactly as
// cross products in 128 bits; equal ratios -> smaller (a, b, ea, eb).
__device__ __forceinline__ bool plan_better(const PlanCandidate& x, const PlanCandidate& y) {
  if (x.ea < 0) return false;
  if (y.ea < 0) return true;
  const unsigned __int128 l = static_cast<unsigned __int128>(static_cast<unsigned long long>(x.benefit)) * y.cost;
  const unsigned __int128 r = static_cast<unsigned __int128>(static_cast<unsigned long long>(y.benefit)) * x.cost;
  if (l != r) return l > r;
  if (x.a != y.a) return x.a < y.a;
  if (x.b != y.b) return x.b < y.b;
  if (x.ea != y.ea) return x.ea < y.ea;
  return x.eb < y.eb;
}

__device__ __forceinline__ unsigned long long plan_cost_ns(const PlanParams& p, int cls, int ea, int eb) {
  if (p.expert_bytes_table == nullptr) return p.uniform_cost_ns[cls];
  const unsigned __int128 bytes = static_cast<unsigned __int128>(p.expert_bytes_table[ea]) + p.expert_bytes_table[eb];
  const unsigned __int128 fs = bytes * p.fs_per_byte[cls];
  unsigned __int128 ns = (fs + 999999u) / 1000000u + p.alpha_ns[cls];
  if (ns > 0xFFFFFFFFFFFFFFFFull) ns = 0xFFFFFFFFFFFFFFFFull;
  const unsigned long long c = static_cast<unsigned long long>(ns);
  return c < 1 ? 1 : c;
}

// Expert e's slot under the placement as given: into shared memory, inverted, checked to be a bijection.
// sh.bad must have been cleared and sh.expert_at filled with -1 beforehand.
__device__ __forceinline__ void plan_place(const PlanParams& p, PlanShared& sh, int e, int s) {
  const bool inside = s >= 0 && s < p.E;
  sh.slot_of[e] = s;
  sh.moved[e] = 0;
  sh.rank_of[e] = static_cast<uint8_t>(inside ? rank_of_slot(p, s) : 0);
  if (!inside || atomicExch(&sh.expert_at[s], e) != -1) sh.bad = 1;
}
__device__ __forceinline__ void plan_place_ranks(const PlanParams& p, PlanShared& sh, int t, int nthreads) {
  for (int r = t; r < p.R; r += nthreads)
    sh.node_of[r] = static_cast<uint8_t>(p.ranks_per_node > 0 ? r / p.ranks_per_node : 0);
}
// The whole placement, by `nthreads` threads (t = 0..nthreads-1); the caller synchronises afterwards.
__device__ __forceinline__ void plan_load_placement(const PlanParams& p, PlanShared& sh, int t, int nthreads) {
  for (int e = t; e < p.E; e += nthreads) plan_place(p, sh, e, p.expert_to_slot[e]);
  plan_place_ranks(p, sh, t, nthreads);
}
__device__ __forceinline__ void plan_clear(PlanShared& sh, int t, int nthreads) {
  if (t == 0) { sh.bad = 0; sh.bad_range = 0; sh.fast = 0; }
  for (int e = t; e < FB_MAX_EXPERTS; e += nthreads) sh.expert_at[e] = -1;
  for (int r = t; r < FB_MAX_RANKS; r += nthreads) sh.load[r] = 0;
}

// The count of expert e arrives (any thread, once per expert, after plan_load_placement and a
// barrier; another barrier follows before the planner warp runs): it goes into the slot word
// of the expert's slot and into its rank's load (Algorithm 1 line 2).
__device__ __forceinline__ void plan_put_count(PlanShared& sh, int e, uint32_t c) {
  sh.cnt[e] = c;
  if (c > FB_MAX_COUNT_SUM) { sh.bad_range = 1; return; }
  if (sh.bad) return;
  sh.slot_cnt[sh.slot_of[e]] = slot_word(c, e);
  atomicAdd(&sh.load[sh.rank_of[e]], c);
}

// The same by the thread that has placed the expert (slot: its slot as given), with no barrier in between.
__device__ __forceinline__ void plan_put_count_at(PlanShared& sh, int e, int slot, uint32_t c, int E) {
  sh.cnt[e] = c;
  if (c > FB_MAX_COUNT_SUM) { sh.bad_range = 1; return; }
  if (slot < 0 || slot >= E) return;
  sh.slot_cnt[slot] = slot_word(c, e);
  atomicAdd(&sh.load[sh.rank_of[e]], c);
}

// The new placement (called by all those threads after the planner warp is done and a
// barrier): slot s holds the expert its slot word names (fast loop) or expert_at[s].  An
// unusable input keeps the placement as given.
__device__ __forceinline__ void plan_write_placement(const PlanParams& p, PlanShared& sh, int t, int nthreads) {
  if (sh.bad || sh.bad_range) {
    for (int e = t; e < p.E; e += nthreads) p.expert_to_slot_out[e] = p.expert_to_slot[e];
  } else if (sh.fast) {
    for (int sl = t; sl < p.E; sl += nthreads) p.expert_to_slot_out[sh.slot_cnt[sl] & 0xffu] = sl;
  } else {
    for (int sl = t; sl < p.E; sl += nthreads) p.expert_to_slot_out[sh.expert_at[sl]] = sl;
  }
}

// Greedy loop specialised for the common case: one cost per link class (no per-expert
// size table).  m experts per rank, m * m candidate pairs per iteration.  One warp runs alone here,
// so what counts is the length of the dependent instruction chain of an iteration.
//
// All pairs of an iteration have the same cost, so the largest benefit / cost is the largest
// benefit.  With d tokens moved from the heavy rank (load La) to the light one (Lb), D = La - Lb and
// v = |2 d - D|: the larger of the two new loads is (La + Lb + v) / 2 and d (D - d) = (D^2 - v^2) / 4, so
//     gamma_den (Phi(L) - Phi(L')) = gamma_den (La - max((La + Lb + v) / 2, M2)) + gamma_num (D^2 - v^2) / 2
// (M2: largest load of the other ranks) falls with v - strictly when gamma_num > 0; when it is 0, it is
// constant up to v = 2 M2 - La - Lb.  A pair is useful exactly if v < D (0 < d < D), and with
// gamma_num = 0 also M2 < La, which the same comparison tests.  The best pair is therefore the one
// with the smallest v (clamped from below when gamma_num = 0), ties to the smallest pair.
// A moved expert counts as 2^22 tokens (kSlotMoved): paired with an unmoved one v is 2^21 or more, beyond any D that it
// could be less than, with a moved one it is D, so no candidate has to be tested - only the smallest v is, against D.
//
// Lane l tries expert slot l / g of the heavy rank with kPerLane slots of the light one, g lanes per
// heavy slot; slots beyond m repeat the last one (the same pair twice in a lane changes nothing; lanes with nothing
// but repeats stand aside).  kPerLane == 0: more
// than 16 experts per rank, lane l takes the heavy slots l, l + 32, ... with every light one (20 experts per
// rank, 4 tokens: layer step 63 us with the general loop below, 22 with this one).  A lane keeps the
// packed (load, rank) keys of its two ranks.
//
// What an iteration waits for: the slot words, a few operations, and two warp reductions, one over v and one over the
// pair, the sign of 2 d - D and the lane - d follows from v and the sign in every lane.  The frontier of the next iteration is
// the larger (smaller) of the two new loads and of the other ranks' largest (smallest), which is reduced meanwhile.
// One branch per iteration: each costs as much as a reduction (22 cycles) or more, and integer operations
// issue every other cycle from a single warp.  With 16 experts per rank 360 cycles per iteration, with 8 240; with
// branches for "balanced", "no pair", ties and the chosen lane 520 and 355, before that (reductions for the frontier as
// well, a shuffle for d, more operations per slot word) 610 and 390.
// In line in its kernels, with the parameters out of constant memory, everything around the loop takes 600 cycles; as a
// function with a pointer to them it took 1400: layer calls of 8192 tokens, 128 experts 25.9 -> 24.3 us, 40 x 128 16.7 ->
// 15.3, 1733 x 256 30.7 -> 29.6.
// kBooks: two cost classes, or per-rank or per-link budgets that can bind.  Otherwise the budgets allow
// a fixed number of swaps (swap_cap) and the loop keeps no books at all.
template <int kPerLane, bool kBooks>
__device__ __forceinline__ uint32_t plan_loop_uniform(const PlanParams& p, PlanShared& sh, int lane,
                                                      int& L0, int& L1, bool write) {
  const int m = p.per_rank;
  const uint32_t full = 0xffffffffu;
  constexpr uint32_t kNone = 0xffffffffu, kNoPair = (1u << 24) - 1;
  constexpr int kNarrow = kPerLane == 0 ? 1 : kPerLane;
  constexpr int g = kPerLane == 8 ? 2 : (kPerLane == 2 ? 4 : 8);     // m <= 16, <= 8, <= 4
  const int ia = min(lane / g, m - 1), j0 = (lane % g) * kNarrow;
  const bool whole = m == g * kNarrow;                            // the lane's light slots are contiguous and exist
  const bool aside = kPerLane != 0 && (lane / g >= m || j0 >= m);
  const bool flat = p.gamma_den == 0 || p.gamma_num == 0;
  const uint32_t tau = p.tau_tokens, max_swaps = kBooks ? p.max_swaps : p.swap_cap;
  // frontier keys (lowest index on ties): max of load << 6 | (63 - rank), min of load << 6 | rank - the same but for
  // the six bits of the rank, which are the other's complement
  const uint32_t none0 = L0 >= 0 ? 0u : kNone, none1 = L1 >= 0 ? 0u : kNone;      // no such rank
  uint32_t h0 = L0 >= 0 ? (static_cast<uint32_t>(L0) << 6 | static_cast<uint32_t>(63 - lane)) : 0u;
  uint32_t h1 = L1 >= 0 ? (static_cast<uint32_t>(L1) << 6 | static_cast<uint32_t>(31 - lane)) : 0u;
  // books
  uint32_t my_links[4] = {kNone, kNone, kNone, kNone};            // lane i keeps the links of swaps i, i+32, ...
  unsigned long long global_spent = 0;
  uint32_t n = 0;
  uint32_t hi_key = __reduce_max_sync(full, max(h0, h1));
  uint32_t lo_key = __reduce_min_sync(full, min(h0 ^ 63u | none0, h1 ^ 63u | none1));
  while (n < max_swaps) {
    const int a = 63 - static_cast<int>(hi_key & 63u), b = static_cast<int>(lo_key & 63u);
    const int La = static_cast<int>(hi_key >> 6), Lb = static_cast<int>(lo_key >> 6);
    const int D = La - Lb;
    const int base_a = a * m, base_b = b * m;
    uint32_t wa = 0, wb[kNarrow];                                 // slot words: twice the count, expert
    if constexpr (kPerLane != 0) {
      wa = sh.slot_cnt[base_a + ia];
      if (kPerLane == 8 && whole) {
#pragma unroll
        for (int t = 0; t < kNarrow; t += 4) {
          const uint4 q = *reinterpret_cast<const uint4*>(&sh.slot_cnt[base_b + j0 + t]);
          wb[t] = q.x; wb[(t + 1) % kNarrow] = q.y; wb[(t + 2) % kNarrow] = q.z; wb[(t + 3) % kNarrow] = q.w;
        }
      } else {
#pragma unroll
        for (int t = 0; t < kNarrow; ++t) wb[t] = sh.slot_cnt[base_b + min(j0 + t, m - 1)];
      }
    }
    bool stop = static_cast<uint32_t>(D) <= tau;                  // (the same in all lanes, as everything that ends the loop)
    unsigned long long c_ns = 0, rs_a = 0, rs_b = 0;
    uint32_t lkey = 0;
    if (kBooks) {
      // the cost is the same for every pair of this iteration
      rs_a = sh.rank_spent[a]; rs_b = sh.rank_spent[b];
      const int node_a = sh.node_of[a], node_b = sh.node_of[b];
      const int cls = node_a == node_b ? 0 : 1;
      c_ns = p.uniform_cost_ns[cls];
      // link: the unordered rank pair inside a node, the unordered node pair across nodes
      const int ka = cls ? node_a : a, kb = cls ? node_b : b;
      lkey = static_cast<uint32_t>(cls) << 16 | static_cast<uint32_t>(ka < kb ? ka : kb) << 8 |
             static_cast<uint32_t>(ka < kb ? kb : ka);
      stop = stop || (p.global_ns != FB_BUDGET_OFF && (c_ns > p.global_ns || global_spent > p.global_ns - c_ns));
      const unsigned long long rs = rs_a > rs_b ? rs_a : rs_b;
      stop = stop || (p.rank_ns != FB_BUDGET_OFF && (c_ns > p.rank_ns || rs > p.rank_ns - c_ns));
      if (p.link_ns != FB_BUDGET_OFF) {
        // A link is only ever charged one cost (its class's), so its budget is a swap count.
        uint32_t used = 0;                                       // swaps already charged to this link
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (n > 32u * q) used += __popc(__ballot_sync(full, my_links[q] == lkey));    // n is the same in all lanes
        stop = stop || used >= p.uniform_link_cap[cls];
      }
    }
    // the other ranks' largest and smallest load
    const bool in0 = lane == a || lane == b, in1 = lane + 32 == a || lane + 32 == b;
    const uint32_t hi_rest = __reduce_max_sync(full, max(in0 ? 0u : h0, in1 ? 0u : h1));
    const uint32_t lo_rest = __reduce_min_sync(full, min(in0 ? kNone : h0 ^ 63u | none0, in1 ? kNone : h1 ^ 63u | none1));
    const int v_floor = flat ? 2 * static_cast<int>(hi_rest >> 6) - La - Lb : 0;
    // ---- smallest v of this lane, ties -> smallest pair; where its experts are, and 2 d - D
    uint32_t mine = kNoPair, pair = 0;
    int sa = 0, sb = 0, off = 0;
    if constexpr (kPerLane != 0) {
      const int y = static_cast<int>(wa >> 8) - D;
      uint32_t key[kNarrow];
#pragma unroll
      for (int t = 0; t < kNarrow; ++t)                           // v << 8 | expert of the light rank
        key[t] = __byte_perm(static_cast<uint32_t>(abs(y - static_cast<int>(wb[t] >> 8))), wb[t], 0x2104);
      if (flat) {
#pragma unroll
        for (int t = 0; t < kNarrow; ++t)
          key[t] = __byte_perm(static_cast<uint32_t>(max(static_cast<int>(key[t] >> 8), v_floor)), wb[t], 0x2104);
      }
      uint32_t best = key[0];
      if constexpr (kNarrow == 8) best = __vimin3_u32(__vimin3_u32(key[0], key[1], key[2]), __vimin3_u32(key[3], key[4], key[5]),
                                                      min(key[6], key[7]));
      else if constexpr (kNarrow == 2) best = min(key[0], key[1]);
      mine = aside ? kNoPair : best >> 8;
      pair = (wa & 0xffu) << 8 | (best & 0xffu);
      sa = base_a + ia;
      uint32_t w_best = wb[0];
      sb = base_b + min(j0, m - 1);
#pragma unroll
      for (int t = kNarrow - 1; t > 0; --t)
        if (key[t] == best) { sb = base_b + min(j0 + t, m - 1); w_best = wb[t]; }
      off = y - static_cast<int>(w_best >> 8);
    } else {
      for (int i = lane; i < m; i += 32) {
        const uint32_t wi = sh.slot_cnt[base_a + i];
        const int y = static_cast<int>(wi >> 8) - D;
        for (int jj = 0; jj < m; jj += 8) {
          uint32_t wj[8];
#pragma unroll
          for (int t = 0; t < 8; ++t) wj[t] = sh.slot_cnt[base_b + min(jj + t, m - 1)];
#pragma unroll
          for (int t = 0; t < 8; ++t) {
            const int o = y - static_cast<int>(wj[t] >> 8);
            const uint32_t v = static_cast<uint32_t>(max(abs(o), v_floor));
            const uint32_t pr = (wi & 0xffu) << 8 | (wj[t] & 0xffu);
            if (v < mine || (v == mine && pr < pair)) {
              mine = v; pair = pr; sa = base_a + i; sb = base_b + min(jj + t, m - 1);
              off = o;
            }
          }
        }
      }
    }
    const uint32_t sign_lane = (off < 0 ? 32u : 0u) | static_cast<uint32_t>(lane);
    const uint32_t top = __reduce_min_sync(full, mine);
    const uint32_t win = __reduce_min_sync(full, mine == top ? pair << 6 | sign_lane : kNone);
    if (stop || top >= static_cast<uint32_t>(D)) break;           // Algorithm 1 lines 6-7
    const int src = static_cast<int>(win & 31u);
    // tokens moved a -> b, in the place of a load: (D + off) / 2 of the chosen lane
    const uint32_t moved = static_cast<uint32_t>(flat ? __shfl_sync(full, D + off, src)
                                                 : D + ((win & 32u) != 0 ? -static_cast<int>(top) : static_cast<int>(top))) << 5;
    // The two experts trade slots.  The accepted swap stays in shared memory until the loop is over (ranks and expert ids
    // are below 256: one word; link_key is otherwise unused on this path): a global store here would be waited for at the
    // warp barrier below, once per iteration.
    const uint32_t chosen = lane == src ? 1u : 0u;
    st_shared_if(chosen, smem_u32(&sh.slot_cnt[sa]), slot_word(kSlotMoved, static_cast<int>(pair & 0xffu)));
    st_shared_if(chosen, smem_u32(&sh.slot_cnt[sb]), slot_word(kSlotMoved, static_cast<int>(pair >> 8)));
    st_shared_if(chosen, smem_u32(&sh.link_key[n]), static_cast<uint32_t>(a) << 24 | static_cast<uint32_t>(b) << 16 | pair);
    if (kBooks && chosen != 0) { sh.rank_spent[a] = rs_a + c_ns; sh.rank_spent[b] = rs_b + c_ns; }
    if (in0) h0 += lane == a ? 0u - moved : moved;
    if (in1) h1 += lane + 32 == a ? 0u - moved : moved;
    const uint32_t new_a = hi_key - moved, new_b = lo_key + moved;
    hi_key = __vimax3_u32(hi_rest, new_a, new_b ^ 63u);
    lo_key = __vimin3_u32(lo_rest, new_a ^ 63u, new_b);
    if (kBooks) {
      if (static_cast<int>(n & 31u) == lane) {
#pragma unroll
        for (int q = 0; q < 4; ++q) if (static_cast<int>(n >> 5) == q) my_links[q] = lkey;
      }
      global_spent += c_ns;
    }
    ++n;
    __syncwarp();                                                 // the next iteration reads what the winner wrote
  }
  if (L0 >= 0) L0 = static_cast<int>(h0 >> 6);
  if (L1 >= 0) L1 = static_cast<int>(h1 >> 6);
  __syncwarp();
  for (uint32_t i = lane; write && i < n; i += 32) {              // the plan, in order of acceptance
    const uint32_t w = sh.link_key[i];
    fb_swap sw;
    sw.src_rank = static_cast<int32_t>(w >> 24); sw.dst_rank = static_cast<int32_t>((w >> 16) & 0xffu);
    sw.expert_src = static_cast<int32_t>((w >> 8) & 0xffu); sw.expert_dst = static_cast<int32_t>(w & 0xffu);
    p.swaps[i] = sw;
  }
  return n;
}

// Which plans the fast loop cannot serve (host and device agree on this test).
__host__ __device__ inline bool plan_needs_general_loop(const PlanParams& p) {
  return p.expert_bytes_table != nullptr || p.mode != FB_PLAN_LOOP;
}

// The general greedy loop: per-expert sizes or a planner variant (the one-pass sweep of the ordering paragraph, a widened frontier).  Plain and slow;
// a function of its own so that its registers and spills stay out of the common path.
// L0 / L1: this lane's rank loads (ranks lane and lane + 32, -1 if absent).
__device__ __noinline__ void plan_loop_general(const PlanParams& p, PlanShared& sh, int lane, long long L0,
                                               long long L1) {
  const int E = p.E, R = p.R, m = E / R;
  const uint32_t full = 0xffffffffu;
  const long long gnum = p.gamma_den ? p.gamma_num : 0;
  const long long gden = p.gamma_den ? p.gamma_den : 1;
  const int rpn = p.ranks_per_node;
  const bool uniform = p.expert_bytes_table == nullptr;     // one cost per link class
  const bool sweep = p.mode == FB_PLAN_SWEEP;
  int W = p.mode == FB_PLAN_WIDE ? p.frontier_width : 1;
  W = W < 1 ? 1 : (W > kMaxFrontierWidth ? kMaxFrontierWidth : W);
  if (W > R) W = R;
  const int mm = m * m;
  unsigned long long global_spent = 0;
  uint32_t n = 0;
  // the sweep scores every pair once, against the frontier and the loads of the placement as given
  int top[kMaxFrontierWidth], bot[kMaxFrontierWidth];
  long long Ltop[kMaxFrontierWidth], Lbot[kMaxFrontierWidth], other_max[kMaxFrontierWidth * kMaxFrontierWidth];
  while (n < p.max_swaps) {
    if (!sweep || n == 0) {
      // The W most and the W least loaded ranks, lowest index on ties, by repeated extraction.
      // Loads are below 2^22, so (load, rank) packs into 32 bits: max of load<<6 | (63 - rank),
      // min of load<<6 | rank.
      unsigned long long taken_hi = 0, taken_lo = 0;
#pragma unroll
      for (int w = 0; w < kMaxFrontierWidth; ++w) {
        if (w < W) {
          const bool f0 = L0 >= 0 && !((taken_hi >> lane) & 1ull), f1 = L1 >= 0 && !((taken_hi >> (lane + 32)) & 1ull);
          const uint32_t h0 = f0 ? (static_cast<uint32_t>(L0) << 6 | static_cast<uint32_t>(63 - lane)) : 0u;
          const uint32_t h1 = f1 ? (static_cast<uint32_t>(L1) << 6 | static_cast<uint32_t>(31 - lane)) : 0u;
          const uint32_t hi_key = __reduce_max_sync(full, h0 > h1 ? h0 : h1);
          top[w] = 63 - static_cast<int>(hi_key & 63u);
          Ltop[w] = hi_key >> 6;
          taken_hi |= 1ull << top[w];
          const bool g0 = L0 >= 0 && !((taken_lo >> lane) & 1ull), g1 = L1 >= 0 && !((taken_lo >> (lane + 32)) & 1ull);
          const uint32_t l0 = g0 ? (static_cast<uint32_t>(L0) << 6 | static_cast<uint32_t>(lane)) : 0xffffffffu;
          const uint32_t l1 = g1 ? (static_cast<uint32_t>(L1) << 6 | static_cast<uint32_t>(lane + 32)) : 0xffffffffu;
          const uint32_t lo_key = __reduce_min_sync(full, l0 < l1 ? l0 : l1);
          bot[w] = static_cast<int>(lo_key & 63u);
          Lbot[w] = lo_key >> 6;
          taken_lo |= 1ull << bot[w];
        }
      }
      // largest load among the ranks other than the two of a pair
#pragma unroll
      for (int wa = 0; wa < kMaxFrontierWidth; ++wa)
#pragma unroll
        for (int wb = 0; wb < kMaxFrontierWidth; ++wb)
          if (wa < W && wb < W) {
            const int a = top[wa], b = bot[wb];
            uint32_t o = 0;
            if (lane != a && lane != b && L0 > 0) o = static_cast<uint32_t>(L0);
            if (lane + 32 != a && lane + 32 != b && L1 > static_cast<long long>(o)) o = static_cast<uint32_t>(L1);
            other_max[wa * kMaxFrontierWidth + wb] = __reduce_max_sync(full, o);
          }
    }
    if (Ltop[0] - Lbot[0] <= static_cast<long long>(p.tau_tokens)) break;
    const long long M = Ltop[0];                                  // the maximum rank load
    PlanCandidate best;
    best.benefit = 0; best.cost = 1; best.a = -1; best.b = -1; best.ea = -1; best.eb = -1;
#pragma unroll
    for (int wa = 0; wa < kMaxFrontierWidth; ++wa) {
#pragma unroll
      for (int wb = 0; wb < kMaxFrontierWidth; ++wb) {
        if (wa >= W || wb >= W) continue;
        const int a = top[wa], b = bot[wb];
        const long long La = Ltop[wa], Lb = Lbot[wb];
        if (a == b || La <= Lb) continue;                         // a source carries strictly more than its destination
        const long long O = other_max[wa * kMaxFrontierWidth + wb];
        const int cls = (rpn <= 0 || a / rpn == b / rpn) ? 0 : 1;
        const int lo = a < b ? a : b, hi = a < b ? b : a;
        const uint32_t lkey = cls == 0 ? (static_cast<uint32_t>(lo) << 8 | static_cast<uint32_t>(hi))
                                       : (0x10000u | static_cast<uint32_t>(lo / rpn) << 8 | static_cast<uint32_t>(hi / rpn));
        unsigned long long link_spent = 0;
        if (p.link_ns != FB_BUDGET_OFF)
          for (uint32_t i = 0; i < n; ++i)
            if (sh.link_key[i] == lkey) link_spent += sh.link_cost[i];
        const unsigned long long rs_a = sh.rank_spent[a], rs_b = sh.rank_spent[b];
        const unsigned long long rank_spent = rs_a > rs_b ? rs_a : rs_b;
        const long long D = La - Lb;
        for (int c = lane; c < mm; c += 32) {
          const int ea = sh.expert_at[a * m + c / m];
          const int eb = sh.expert_at[b * m + c % m];
          if (sh.moved[ea] || sh.moved[eb]) continue;
          const long long dlt = static_cast<long long>(sh.cnt[ea]) - static_cast<long long>(sh.cnt[eb]);   // tokens moved a -> b
          long long Mn = La - dlt;                                // Eq. 6
          if (Lb + dlt > Mn) Mn = Lb + dlt;                       // Eq. 7
          if (O > Mn) Mn = O;
          // gamma_den * (Phi(L) - Phi(L')): the mean is unchanged by a swap, so the
          // variance term reduces to 2 dlt (La - Lb - dlt).
          const long long benefit = gden * (M - Mn) + 2 * gnum * (dlt * (D - dlt));
          if (benefit <= 0) continue;
          PlanCandidate cand;
          cand.benefit = benefit;
          cand.a = a; cand.b = b; cand.ea = ea; cand.eb = eb;
          cand.cost = uniform ? p.uniform_cost_ns[cls] : plan_cost_ns(p, cls, ea, eb);   // Eq. 9
          if (p.global_ns != FB_BUDGET_OFF && (cand.cost > p.global_ns || global_spent > p.global_ns - cand.cost)) continue;
          if (p.rank_ns != FB_BUDGET_OFF && (cand.cost > p.rank_ns || rank_spent > p.rank_ns - cand.cost)) continue;
          if (p.link_ns != FB_BUDGET_OFF && (cand.cost > p.link_ns || link_spent > p.link_ns - cand.cost)) continue;
          if (plan_better(cand, best)) best = cand;
        }
      }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      PlanCandidate o;
      o.benefit = __shfl_xor_sync(full, best.benefit, off);
      o.cost = __shfl_xor_sync(full, best.cost, off);
      o.a = __shfl_xor_sync(full, best.a, off);
      o.b = __shfl_xor_sync(full, best.b, off);
      o.ea = __shfl_xor_sync(full, best.ea, off);
      o.eb = __shfl_xor_sync(full, best.eb, off);
      if (plan_better(o, best)) best = o;
    }
    if (best.ea < 0) break;                                     // Algorithm 1 lines 6-7
    const int a = best.a, b = best.b;
    const long long dlt = static_cast<long long>(sh.cnt[best.ea]) - static_cast<long long>(sh.cnt[best.eb]);
    const int cls = (rpn <= 0 || a / rpn == b / rpn) ? 0 : 1;
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    const uint32_t lkey = cls == 0 ? (static_cast<uint32_t>(lo) << 8 | static_cast<uint32_t>(hi))
                                   : (0x10000u | static_cast<uint32_t>(lo / rpn) << 8 | static_cast<uint32_t>(hi / rpn));
    __syncwarp();                                               // all lanes are done reading the tables
    if (lane == 0) {
      const int sa = sh.slot_of[best.ea], sb = sh.slot_of[best.eb];
      sh.slot_of[best.ea] = sb; sh.slot_of[best.eb] = sa;
      sh.expert_at[sa] = best.eb; sh.expert_at[sb] = best.ea;
      sh.moved[best.ea] = 1; sh.moved[best.eb] = 1;
      sh.rank_spent[a] += best.cost; sh.rank_spent[b] += best.cost;
      sh.link_key[n] = lkey; sh.link_cost[n] = best.cost;
      fb_swap sw; sw.src_rank = a; sw.dst_rank = b; sw.expert_src = best.ea; sw.expert_dst = best.eb;
      p.swaps[n] = sw;
    }
    if (lane == a) L0 -= dlt;
    if (lane + 32 == a) L1 -= dlt;
    if (lane == b) L0 += dlt;
    if (lane + 32 == b) L1 += dlt;
    global_spent += best.cost;
    ++n;
    __syncwarp();
  }
  if (lane == 0) *p.n_swaps = static_cast<int32_t>(n);
  if (lane < R) p.load_after[lane] = static_cast<uint32_t>(L0);
  if (lane + 32 < R) p.load_after[lane + 32] = static_cast<uint32_t>(L1);
}

// The planner, run by ONE warp (all 32 lanes) once plan_load_placement has filled the
// placement arrays and plan_put_count has turned the count vector into counts per slot.  A single
// warp keeps the rank loads in registers (lane r holds ranks r and r + 32) and needs no block barrier.  Writes the swaps, their number and the rank loads
// before and after; the new placement is written afterwards by plan_write_placement.
// kGeneral: the instance carries the general loop as well.  Only a planner kernel's does (the host launches it behind
// the router kernel when a plan needs the general loop - see plan_needs_general_loop): the general loop's registers
// and code would otherwise weigh on every other kernel that plans.
// write: whether this warp's results go to global memory (several blocks may replay a plan, see the
// dispatch index); only for instances without the general loop.
// In line: its parameters come out of constant memory that way (see plan_loop_uniform).
template <bool kGeneral>
__device__ __forceinline__ void plan_swaps_warp(const PlanParams& p, PlanShared& sh, int lane, int* status,
                                                bool write = true, unsigned long long* stamps = nullptr) {
  const int R = p.R, m = p.per_rank;
  const uint32_t full = 0xffffffffu;
  __syncwarp();
  FB_PLAN_STAMP(18);
  // ---- rank loads (Algorithm 1 line 2), formed by plan_put_count: lane holds L[lane] and
  // L[lane + 32]; their sum is checked against the planner's range
  const unsigned long long s0 = lane < R ? sh.load[lane] : 0u, s1 = lane + 32 < R ? sh.load[lane + 32] : 0u;
  const uint32_t total = __reduce_add_sync(full, static_cast<uint32_t>(s0 + s1));   // at most 256 counts of <= 2^21 each
  int bad = sh.bad ? 1 : ((sh.bad_range || total > FB_MAX_COUNT_SUM) ? 2 : 0);
  if (bad) {
    // Unusable input: report it, keep the placement as given, empty plan.
    if (lane == 0 && write) {
      atomicCAS(status, 0, bad == 1 ? FB_ERR_BAD_PLACEMENT : FB_ERR_RANGE);
      *p.n_swaps = 0;
    }
    if (lane == 0) sh.bad_range = 1;             // plan_write_placement copies the input placement
    for (int r = lane; write && r < R; r += 32) { p.load_before[r] = 0; p.load_after[r] = 0; }
    return;
  }
  long long L0 = -1, L1 = -1;                  // -1 marks "no such rank"
  if (lane < R) {
    L0 = static_cast<long long>(s0);
    if (write) p.load_before[lane] = static_cast<uint32_t>(s0);
    sh.rank_spent[lane] = 0;
  }
  if (lane + 32 < R) {
    L1 = static_cast<long long>(s1);
    if (write) p.load_before[lane + 32] = static_cast<uint32_t>(s1);
    sh.rank_spent[lane + 32] = 0;
  }
  __syncwarp();
  FB_PLAN_STAMP(19);

  if (!plan_needs_general_loop(p)) {
    int l0 = static_cast<int>(L0), l1 = static_cast<int>(L1);
    uint32_t n_fast;
    if (lane == 0) sh.fast = 1;
    if (!p.books)
      n_fast = m <= 4 ? plan_loop_uniform<1, false>(p, sh, lane, l0, l1, write)
               : m <= 8 ? plan_loop_uniform<2, false>(p, sh, lane, l0, l1, write)
               : m <= 16 ? plan_loop_uniform<8, false>(p, sh, lane, l0, l1, write)
                         : plan_loop_uniform<0, false>(p, sh, lane, l0, l1, write);
    else
      n_fast = m <= 4 ? plan_loop_uniform<1, true>(p, sh, lane, l0, l1, write)
               : m <= 8 ? plan_loop_uniform<2, true>(p, sh, lane, l0, l1, write)
               : m <= 16 ? plan_loop_uniform<8, true>(p, sh, lane, l0, l1, write)
                         : plan_loop_uniform<0, true>(p, sh, lane, l0, l1, write);
    FB_PLAN_STAMP(20);
    if (lane == 0 && write) *p.n_swaps = static_cast<int32_t>(n_fast);
    if (lane < R && write) p.load_after[lane] = static_cast<uint32_t>(l0);
    if (lane + 32 < R && write) p.load_after[lane + 32] = static_cast<uint32_t>(l1);
    return;
  }
  if constexpr (kGeneral) {
    plan_loop_general(p, sh, lane, L0, L1);
  } else {
    // not reachable when the host follows plan_needs_general_loop; an empty plan otherwise
    if (lane == 0) *p.n_swaps = 0;
    if (lane < R) p.load_after[lane] = static_cast<uint32_t>(L0);
    if (lane + 32 < R) p.load_after[lane + 32] = static_cast<uint32_t>(L1);
  }
}

// The same as a function of its own, for the router kernels: only launches of more tiles than the GPU holds at once plan there.
// In line and apart, calls that do not reach it: layer 40 tokens, 128 experts 13.1 and 12.9 us, 512 x 8 9.9 and 9.7, 8192 x 128
// 20.2 and 20.3; that do: layer 131072 x 128 182.0 and 180.9 (spread 1.5), prediction and plan 24000 x 256 93.6 and 94.1
// (spread 1), 20000 x 128 33.5 and 34.7.
__device__ __noinline__ void plan_swaps_apart(const PlanParams& p, PlanShared& sh, int lane, int* status,
                                              unsigned long long* stamps) {
  plan_swaps_warp<false>(p, sh, lane, status, true, stamps);
}

}  // namespace fb
