// Fused router kernel for calls with few tiles and for gates that the ranking selection does not
// serve: logits = x W^T (+ b) as in fb_router_kernel, then a WARP per token row for gating and top-k.
//
// Work split.  Two blocks of a cluster (a pair) compute a tile pair: 256 token rows x all N = pad16(E)
// expert columns with one cta_group::2 MMA; each loads its own 128 rows of x and half of the W tile.
//   * Few tile pairs: a cluster of 2 J blocks (J = 2 .. 8 pairs) works on ONE tile pair.  Pair j
//     accumulates the j-th piece of the k-range; the J partial tiles meet through distributed shared
//     memory, and each block finishes about 128 / J of its rows.  Both the stream of operands and the
//     selection work are then spread over J times as many SMs, and nothing but a cluster barrier lies
//     between the two.
//   * More tile pairs than pairs fit on the GPU: every pair walks a strided list of tile pairs, and
//     the selection of one tile runs while the tensor cores already work on the next one.
// Warp roles as in fb_router_kernel.
//
// Epilogue.  The 16 epilogue warps copy the sums from tensor memory (one row per thread) to shared
// memory row by row ("staging", rows padded by 16 bytes: conflict-free both ways), and from there on a
// warp owns a token row: the lanes hold its keys in registers, group scores and bounds are formed by a
// few shuffles and warp reductions, the keys that can still enter the top-k (about 10 of 256) are
// compacted into a short list and ranked there.  Any gate fits the same code, no barrier separates the
// steps, and a tile cut into J row slices keeps the warps busy.  It costs more instructions per row than
// the ranking selection with one row per thread where that one has whole tiles to itself (16384 rows x 256
// columns, d = 512, sigmoid groups: 21.6 against 18.1 us per prediction pass; 128 columns, softmax: 16.0
// against 15.3), so those launches stay there; against the insertion code that other gates had before it
// is faster throughout (64 experts, sigmoid without groups: 25.9 -> 14.9 us).
#pragma once
#include <stddef.h>

#include "fb_router.cuh"

namespace fb {

// How a gate's columns lie over the lanes (host).  Returns the number of columns a lane holds, rounded up
// to a power of two (the kernel instance), at most 16.
inline int gate_layout(int E, int gate, int n_group, int topk_group, RouterParams* p) {
  const bool restricted = gate != FB_GATE_SOFTMAX_TOPK && topk_group < n_group;
  const int groups = restricted ? n_group : 1, gs = E / groups;
  int lpg = 1;
  while (lpg * 2 * groups <= 32) lpg *= 2;
  const int per_lane = (gs + lpg - 1) / lpg;
  int cpl = 1;
  while (cpl < per_lane) cpl *= 2;
  p->groups = groups;
  p->group_size = gs;
  p->keep_groups = restricted ? topk_group : 1;
  p->lanes_per_group = lpg;
  // one group, or groups that start on a vector: round the lane's share up so that it is whole vectors
  p->vector_load = (groups == 1 || gs % (cpl < 4 ? cpl : 4) == 0) ? 1 : 0;
  p->cols_per_lane = p->vector_load ? cpl : per_lane;
  p->two_vectors = (cpl == 8 && p->vector_load && E > 128) ? 1 : 0;      // (only rows above 128 columns are padded to 256 words)
  p->ragged = groups * lpg * cpl != E || groups * lpg != 32 ? 1 : 0;
  return cpl;
}

// Staged logits: rows of N + 4 floats.  A warp writes 32 rows of one 16-byte column group at a time, 8
// rows per wavefront: N is a multiple of 16, so the row stride is 4 or 20 words modulo 32 and those 8 rows
// hit all 32 banks once.
// Rows of more than 128 columns are padded to 256: lanes with eight columns each hold two vectors, which
// are stored 128 words apart (all lanes' first vectors, then all second ones), so that a warp's loads are
// contiguous - for rows of other blocks, read over the cluster's network, 512-byte pieces instead of
// 16-byte ones (1733 tokens, 256 experts, four pairs per tile: the selection took 13 us with the latter).
__host__ __device__ constexpr int staging_stride(int N) { return (N > 128 ? 256 : N) + 4; }
constexpr int kListStride = kCandCap + 12;     // + the last lane's columns, rounded up (never read); 12 banks apart for two rows
struct RowScratch {                    // one per epilogue warp
  alignas(16) float cand_key[2][kListStride];  // keys of two rows' candidates in ascending id order; -inf behind the last one
  alignas(16) int32_t cand_id[2][kListStride];
  alignas(16) int2 win[8][FB_MAX_TOPK];        // the rows' top-k in order of rank: key (its bits), expert id
  float row_sum[8];                            // softmax denominators relative to the row's largest key
};
__host__ __device__ constexpr size_t staging_bytes(int rows, int N) {
  return static_cast<size_t>(rows) * staging_stride(N) * 4 + kEpilogueWarps * sizeof(RowScratch);
}

// What a lane needs to know about its columns.
struct LaneColumns {
  int32_t c0, n;                       // first column, number of columns
  int32_t word;                        // where they start in a staged row
  int32_t group;                       // group of its columns (>= groups: an idle lane)
};
__host__ __device__ inline LaneColumns lane_columns(const RouterParams& p, int lane) {
  LaneColumns lc;
  lc.group = lane / p.lanes_per_group;
  const int first = lane % p.lanes_per_group * p.cols_per_lane, left = p.group_size - first;
  lc.n = lc.group >= p.groups || left <= 0 ? 0 : (left < p.cols_per_lane ? left : p.cols_per_lane);
  lc.c0 = lc.n == 0 ? 0 : lc.group * p.group_size + first;
  lc.word = p.two_vectors ? 4 * lane : lc.c0;
  return lc;
}
// Where columns 4 q .. 4 q + 3 lie in a staged row.  (A quad lies in one group and one lane where rows are stored
// as two vectors per lane; groups start on a quad there; padding columns go behind the lanes' words.)
__host__ __device__ inline int quad_word(const RouterParams& p, int q) {
  if (!p.two_vectors) return 4 * q;
  const int in = 4 * q % p.group_size, of_lane = 4 * q / p.group_size * p.lanes_per_group + in / 8;
  return 4 * q < p.E ? in / 4 % 2 * 128 + of_lane * 4 : 256;
}

struct RowsShared {
  uint64_t full_bar[kMaxStages];
  uint64_t empty_bar[kMaxStages];
  // Accumulator sets (of N columns per issuer): one, or two that alternate where a pair walks several
  // tiles, so that the next tile's MMAs need not wait for the drain.
  uint64_t accum_bar[2];                     // per set: both issuers' commits, once per use
  uint64_t tmem_empty_bar[2];                // per set, even block's copy: all epilogue warps of the pair, once per use
  uint64_t staged_bar;                       // the blocks that share this block's tile have staged their sums
  uint32_t tmem_base;
  int32_t abort_flag;
  int32_t is_last;
  int32_t accum_ok;
  int32_t started;                           // the wait for the kernels before this one is over (prefetch_operands)
  int32_t issuer_progress[2];                // where both issuers use a stage: see issuer_turn_wait
  uint16_t quad_word[FB_MAX_EXPERTS / 4];    // where columns 4 q .. 4 q + 3 lie in a staged row
  alignas(16) float logit_bias[FB_MAX_EXPERTS];
  alignas(16) float select_bias[FB_MAX_EXPERTS];
  alignas(16) uint32_t hist[FB_MAX_EXPERTS];
  PlanShared plan;
};

// ---------------------------------------------------------------- selection, one warp per token row
// Plain selection of one row by repeated maximum over keys in shared memory (dropped columns hold
// -inf): the path of rows with more candidates than the list holds, and of rows with equal keys among
// the candidates (the lower expert id wins).  Rare; kept out of line.
__device__ __noinline__ void select_slow(float* keys, int E, int k, int2* win, int lane) {
  for (int r = 0; r < k; ++r) {
    float best = -INFINITY;
    int at = E;
    for (int e = lane; e < E; e += 32)
      if (keys[e] > best) { best = keys[e]; at = e; }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      const float ob = __shfl_xor_sync(0xffffffffu, best, off);
      const int oa = __shfl_xor_sync(0xffffffffu, at, off);
      if (ob > best || (ob == best && oa < at)) { best = ob; at = oa; }
    }
    if (at >= E) {
      // Nothing above -inf is left (masked experts, keys that are no numbers): the other ranks get the lowest ids the
      // row has not named, so that it never names an expert twice.  Fewer than 8 are named: these lie below k <= E.
      if (lane == 0) {
        uint32_t named = 0;
        for (int h = 0; h < r; ++h)
          if (win[h].y < FB_MAX_TOPK) named |= 1u << win[h].y;
        for (int h = r; h < k; ++h) {
          win[h] = make_int2(__float_as_int(-INFINITY), __ffs(~named) - 1);
          named |= 1u << win[h].y;
        }
      }
      break;
    }
    if (lane == 0) { win[r] = make_int2(__float_as_int(best), at); keys[at] = -INFINITY; }
    __syncwarp();
  }
}

// A lane's columns of one staged row of this block / of the block with cluster rank `rank` at the same
// place.  Lanes without columns read valid words all the same; what they read is masked afterwards.
template <int kCpl>
__device__ __forceinline__ void load_columns(float (&z)[kCpl], uint32_t addr, const RouterParams& p, int n) {
  if constexpr (kCpl == 8) {
    if (p.two_vectors) { ld_shared_two_vectors(addr, z); return; }
  }
  if (kCpl == 1 || p.vector_load) {
    ld_shared_floats<kCpl>(addr, z);
  } else {
#pragma unroll
    for (int j = 0; j < kCpl; ++j) z[j] = ld_shared_float(addr + 4 * max(0, min(j, n - 1)));
  }
}
template <int kCpl>
__device__ __forceinline__ void load_columns_of(float (&z)[kCpl], uint32_t addr, uint32_t rank, const RouterParams& p, int n) {
  const uint32_t remote = map_to_cta(addr, rank);
  if constexpr (kCpl == 8) {
    if (p.two_vectors) { ld_cluster_two_vectors(remote, z); return; }
  }
  if (kCpl == 1 || p.vector_load) {
    ld_cluster_floats<kCpl>(remote, z);
  } else {
#pragma unroll
    for (int j = 0; j < kCpl; ++j) z[j] = ld_cluster_float(remote + 4 * max(0, min(j, n - 1)));
  }
}

// r += a > b
__device__ __forceinline__ void count_greater(int& r, float a, float b) {
  asm("{\n.reg .pred p;\nsetp.gt.f32 p, %1, %2;\n@p add.s32 %0, %0, 1;\n}" : "+r"(r) : "f"(a), "f"(b));
}
// key >= bound: key and id to the lists at `slot`, which moves on (predicated, no branch)
__device__ __forceinline__ void append_candidate(uint32_t& slot, float key, float bound, int id) {
  constexpr int kIdOffset = static_cast<int>(offsetof(RowScratch, cand_id) - offsetof(RowScratch, cand_key));
  asm volatile(
      "{\n.reg .pred p;\nsetp.ge.f32 p, %1, %2;\n@p st.shared.f32 [%0], %1;\n@p st.shared.u32 [%0 + %4], %3;\n"
      "@p add.u32 %0, %0, 4;\n}"
      : "+r"(slot) : "f"(key), "f"(bound), "r"(id), "n"(kIdOffset) : "memory");
}

// Softmax denominator of a row relative to its largest key, for weights without renormalisation.
template <int kCpl>
__device__ __forceinline__ float row_exp_sum(const float (&key)[kCpl], float lane_max) {
  const float top = redux_max_f32(lane_max);
  float s = 0.0f;
#pragma unroll
  for (int j = 0; j < kCpl; ++j) s += __expf(key[j] - top);                 // exp(-inf) = 0 for missing columns
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  return s;
}

// The top-k of two staged rows (row_addr: shared-memory address of the first one's first word in this block;
// the J blocks of the cluster whose ranks have my_rank's parity hold one partial sum each at the same place) into
// rows 2 pair and 2 pair + 1 of the scratch's result lists.  row: token index of the first one.
// Two rows at a time because a row's steps are a chain of short dependent ones.
template <int kCpl, bool kSigmoid>
__device__ __forceinline__ void select_two_rows(const RouterParams& p, const LaneColumns& lc, const float (&sb)[kCpl],
                                                const float* logit_bias_s, uint32_t row_addr, uint32_t my_rank,
                                                long long row, float* out_logits, RowScratch& rs, int pair, int lane) {
  const uint32_t full = 0xffffffffu;
  const uint32_t stride = static_cast<uint32_t>(staging_stride(p.N)) * 4u;
  const bool want_sum = !kSigmoid && p.topk_w != nullptr && !p.renorm;
  float key[2][kCpl];
  // ---- logits: the J partial sums, beginning with this block's own.  Which one is added when depends on the
  // row's place in its tile only.  (With all blocks beginning at the same one, its outgoing 16 bytes per
  // cycle served the whole cluster: 475 tokens, 256 experts, eight pairs per tile 25.3 us for prediction and plan
  // and 22.2 in turn.)
  const uint32_t a0 = row_addr + static_cast<uint32_t>(lc.word) * 4u;
  if (p.pieces == 1) {
#pragma unroll
    for (int u = 0; u < 2; ++u) load_columns<kCpl>(key[u], a0 + u * stride, p, lc.n);
  } else {
#pragma unroll
    for (int u = 0; u < 2; ++u) load_columns<kCpl>(key[u], a0 + u * stride, p, lc.n);
    uint32_t from = my_rank;
    // (one, two, three and seven pieces' loads in flight with few columns per lane: 1000 x 128 14.2, 14.2, 14.5, 14.7 us, 40 x 128
    // 13.0 to 13.1, 5 x 128 13.4, 13.1, 13.4, 13.5; with eight columns two and four were 0.6 us slower than one)
#pragma unroll (kCpl >= 8 ? 1 : 2)
    for (int i = 1; i < p.pieces; ++i) {
      float t[2][kCpl];
      from = from + 2 < 2u * p.pieces ? from + 2 : from + 2 - 2u * p.pieces;
#pragma unroll
      for (int u = 0; u < 2; ++u) load_columns_of<kCpl>(t[u], a0 + u * stride, from, p, lc.n);
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int j = 0; j < kCpl; ++j) key[u][j] += t[u][j];
    }
  }
  if (p.logit_bias != nullptr) {
#pragma unroll
    for (int j = 0; j < kCpl; ++j) {
      const float b = logit_bias_s[lc.c0 + max(0, min(j, lc.n - 1))];
      key[0][j] += b;
      key[1][j] += b;
    }
  }
  if (out_logits != nullptr) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int j = 0; j < kCpl; ++j)
        if (j < lc.n && row + u < p.T) out_logits[(row + u) * p.E + lc.c0 + j] = key[u][j];
  }
  // ---- selection keys
  if (kSigmoid) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int j = 0; j < kCpl; ++j) key[u][j] = fb_sigmoid(key[u][j]) + sb[j];
  }
  // Few keys per lane (see below): keys that are no numbers count as -inf, and no number stands for a key that was taken
  // or a column that does not exist - for the latter once group scores and the softmax denominator are formed.
  constexpr bool kFewKeys = kCpl <= 4;
  const float taken = __int_as_float(0x7fffffff);
  const bool mask_later = p.groups > 1 || want_sum;
  if (kFewKeys) {
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int j = 0; j < kCpl; ++j) key[u][j] = fmaxf(key[u][j], -INFINITY);
  }
  if (p.ragged) {
    const float missing = kFewKeys && !mask_later ? taken : -INFINITY;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int j = 0; j < kCpl; ++j) key[u][j] = j < lc.n ? key[u][j] : missing;
  }
  // ---- groups: score = sum of the two largest keys (the only key of a one-expert group); the best
  // keep_groups are kept, a lower-numbered group wins ties
  float bound[2];                                            // lower bound for the k-th key; +inf in a lane of a dropped group
  const bool bound_from_groups = p.groups > 1 && p.keep_groups * (p.group_size >= 2 ? 2 : 1) >= p.k;
  bool kept[2] = {true, true};
  if (p.groups > 1) {
    float m1[2], m2[2];                                      // the lane's, then the group's two largest keys
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (kCpl == 1) {
        m1[u] = key[u][0];
        m2[u] = -INFINITY;
      } else {
        float t1[kCpl / 2 + 1], t2[kCpl / 2 + 1];
#pragma unroll
        for (int j = 0; j < kCpl / 2; ++j) {
          t1[j] = fmaxf(key[u][2 * j], key[u][2 * j + 1]);
          t2[j] = fminf(key[u][2 * j], key[u][2 * j + 1]);
        }
#pragma unroll
        for (int w = kCpl / 4; w >= 1; w >>= 1)
#pragma unroll
          for (int j = 0; j < w; ++j) {
            t2[j] = fmaxf(fmaxf(fminf(t1[j], t1[j + w]), t2[j]), t2[j + w]);
            t1[j] = fmaxf(t1[j], t1[j + w]);
          }
        m1[u] = t1[0];
        m2[u] = t2[0];
      }
    }
    for (int off = 1; off < p.lanes_per_group; off <<= 1) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float o1 = __shfl_xor_sync(full, m1[u], off), o2 = __shfl_xor_sync(full, m2[u], off);
        m2[u] = fmaxf(fmaxf(fminf(m1[u], o1), m2[u]), o2);
        m1[u] = fmaxf(m1[u], o1);
      }
    }
    if (p.group_size == 1) { m2[0] = m1[0]; m2[1] = m1[1]; }     // the smallest known key of the group
    float score[2];
    int rank[2] = {0, 0};
    const bool in_group = lc.group < p.groups;
#pragma unroll
    for (int u = 0; u < 2; ++u) score[u] = in_group ? (p.group_size >= 2 ? m1[u] + m2[u] : m1[u]) : -INFINITY;
    const int lanes = p.groups * p.lanes_per_group;
    int src = lane;
    for (int h = 1; h < p.groups; ++h) {
      src += p.lanes_per_group;
      if (src >= lanes) src -= lanes;
#pragma unroll
      for (int u = 0; u < 2; ++u) count_greater(rank[u], __shfl_sync(full, score[u], src), score[u]);
    }
    const int keep_lanes = p.keep_groups * p.lanes_per_group;
#pragma unroll
    for (int u = 0; u < 2; ++u) kept[u] = in_group && rank[u] < p.keep_groups;
    const uint32_t b0 = __ballot_sync(full, kept[0]), b1 = __ballot_sync(full, kept[1]);
    if (__popc(b0) != keep_lanes || __popc(b1) != keep_lanes) {
      // equal scores (or scores that are no numbers): count again, the lower group first
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        int r = 0;
        for (int g = 0; g < p.groups; ++g) {
          const float os = __shfl_sync(full, score[u], g * p.lanes_per_group);
          r += (os > score[u] || (os == score[u] && g < lc.group)) ? 1 : 0;
        }
        kept[u] = in_group && r < p.keep_groups;
      }
    }
    // the kept groups' best (two) keys are known keys: if there are at least k, the smallest bounds the k-th
    if (bound_from_groups) {
#pragma unroll
      for (int u = 0; u < 2; ++u) bound[u] = redux_min_f32(kept[u] ? m2[u] : INFINITY);
    }
  }
  if (kFewKeys) {
    // Few keys per lane: k rounds of "largest remaining key".  (Compacting the keys above a bound and ranking them, as
    // below, takes k reductions for the bound alone: layer step 40 tokens x 128 experts 18.5 us that way and 17.3 this way,
    // 5003 x 64 25.4 and 24.6, prediction and plan 2729 x 60 16.0 and 14.3.)
    // A lane first puts its keys into descending order, so that a round is one reduction over the lanes' first keys: the lane that
    // holds the largest stores it and moves up, without a branch.  Equal keys in one lane keep their order; if two lanes ever
    // hold the largest, or it is -inf (masked experts, dropped groups, keys that are no numbers, columns that do not exist),
    // the rows are selected once more below, where the lower id is looked for.  Against that form for all rows: layer call
    // 5003 x 64 20.5 -> 18.9 us, 40 x 128 14.5 -> 14.0, 2000 x 60 15.6 -> 15.0, prediction and plan 8192 x 128 19.7 -> 18.3.
    float first[2][kCpl];
    int id[2][kCpl];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
#pragma unroll
      for (int j = 0; j < kCpl; ++j) {
        if (p.groups > 1) key[u][j] = kept[u] ? key[u][j] : -INFINITY;
        first[u][j] = j < lc.n ? key[u][j] : -INFINITY;
        id[u][j] = lc.c0 + j;
      }
#pragma unroll
      for (int pass = 0; pass < kCpl; ++pass)
#pragma unroll
        for (int j = pass & 1; j + 1 < kCpl; j += 2) {
          const bool swap = first[u][j + 1] > first[u][j];
          const float hi = fmaxf(first[u][j], first[u][j + 1]), lo = fminf(first[u][j], first[u][j + 1]);
          const int ih = swap ? id[u][j + 1] : id[u][j], il = swap ? id[u][j] : id[u][j + 1];
          first[u][j] = hi; first[u][j + 1] = lo;
          id[u][j] = ih; id[u][j + 1] = il;
        }
      if (want_sum) {
        const float s = row_exp_sum<kCpl>(key[u], first[u][0]);
        if (lane == 0) rs.row_sum[2 * pair + u] = s;
      }
    }
    uint32_t several[2] = {0, 0};
    float last[2] = {0.0f, 0.0f};
#pragma unroll 1
    for (int r = 0; r < p.k; ++r) {
#pragma unroll
      for (int u = 0; u < 2; ++u) last[u] = redux_max_f32(first[u][0]);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const bool mine = first[u][0] == last[u];
        const uint32_t holders = __ballot_sync(full, mine);
        several[u] |= holders & (holders - 1);
        if (mine) rs.win[2 * pair + u][r] = make_int2(__float_as_int(first[u][0]), id[u][0]);
#pragma unroll
        for (int j = 0; j < kCpl; ++j) {
          first[u][j] = mine ? (j + 1 < kCpl ? first[u][j + 1] : -INFINITY) : first[u][j];
          if (j + 1 < kCpl) id[u][j] = mine ? id[u][j + 1] : id[u][j];
        }
      }
    }
    if ((several[0] | several[1]) == 0 && fminf(last[0], last[1]) > -INFINITY) return;
    // The row behind the last token holds zeros, all equal, and nobody reads what it chose (prediction of 41 tokens, 128
    // experts, into the same buffers 0.8 us longer than of 42 when it was selected again).
    if (row + 1 >= p.T && several[0] == 0 && last[0] > -INFINITY) return;
    // Once more: the lowest lane, and in it the lowest column, has the lowest id on ties.  Keys taken, and columns that do
    // not exist, are no numbers, which no maximum takes up: what is left to take are numbers, -inf for experts that are masked
    // out or in dropped groups, and every row has E >= k of them.
    __syncwarp();
    float lane_max[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      if (p.ragged && mask_later) {
#pragma unroll
        for (int j = 0; j < kCpl; ++j) key[u][j] = j < lc.n ? key[u][j] : taken;
      }
      lane_max[u] = key[u][0];
#pragma unroll
      for (int j = 1; j < kCpl; ++j) lane_max[u] = fmaxf(lane_max[u], key[u][j]);
    }
#pragma unroll 1
    for (int r = 0; r < p.k; ++r) {
      float top[2];
      uint32_t holders[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) top[u] = redux_max_f32(lane_max[u]);
#pragma unroll
      for (int u = 0; u < 2; ++u) holders[u] = __ballot_sync(full, lane_max[u] == top[u]);
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (lane == __ffs(holders[u]) - 1) {
          int at = 0;
#pragma unroll
          for (int j = kCpl - 1; j >= 0; --j) at = key[u][j] == top[u] ? j : at;
          rs.win[2 * pair + u][r] = make_int2(__float_as_int(top[u]), lc.c0 + at);
#pragma unroll
          for (int j = 0; j < kCpl; ++j) key[u][j] = j == at ? taken : key[u][j];
          lane_max[u] = key[u][0];
#pragma unroll
          for (int j = 1; j < kCpl; ++j) lane_max[u] = fmaxf(lane_max[u], key[u][j]);
        }
      }
    }
    return;
  }
  if (!bound_from_groups) {
    // the k-th largest of the (kept) lanes' largest keys
    float lane_max[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      lane_max[u] = key[u][0];
#pragma unroll
      for (int j = 1; j < kCpl; ++j) lane_max[u] = fmaxf(lane_max[u], key[u][j]);
      if (p.groups > 1) lane_max[u] = kept[u] ? lane_max[u] : -INFINITY;
    }
    if (want_sum) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float s = row_exp_sum<kCpl>(key[u], lane_max[u]);
        if (lane == 0) rs.row_sum[2 * pair + u] = s;
      }
    }
#pragma unroll 1
    for (int r = 0; r < p.k; ++r) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        bound[u] = redux_max_f32(lane_max[u]);
        lane_max[u] = lane_max[u] == bound[u] ? -INFINITY : lane_max[u];
      }
    }
  }
  // missing columns and dropped groups never qualify
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    bound[u] = fmaxf(bound[u], -3.402823466e38f);
    if (p.groups > 1) bound[u] = kept[u] ? bound[u] : INFINITY;
  }
  // ---- compact the keys at or above the bound, in ascending id order (lanes hold ascending columns):
  // first every lane's place in the list, then the stores
  const uint32_t below = (1u << lane) - 1u;
  const uint32_t list0 = smem_u32(&rs.cand_key[0][0]);
  int n[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    n[u] = 0;
#pragma unroll
    for (int j = 0; j < kCpl; ++j) n[u] += __popc(__ballot_sync(full, key[u][j] >= bound[u]) & below);
    rs.cand_key[u][lane] = -INFINITY;
  }
  __syncwarp();
  // The last lane starts at most kCandCap entries in and adds at most kCpl: no store leaves the list.
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int last = __shfl_sync(full, n[u], 31);            // candidates before the last lane's
    if (last <= kListStride - (kCpl > 12 ? kCpl : 12)) {     // (the same for the whole warp)
      uint32_t slot = list0 + static_cast<uint32_t>(u * kListStride + n[u]) * 4u;
#pragma unroll
      for (int j = 0; j < kCpl; ++j) append_candidate(slot, key[u][j], bound[u], lc.c0 + j);
      n[u] = __shfl_sync(full, static_cast<int>(slot - list0) / 4 - u * kListStride, 31);
    } else {
      n[u] = kCandCap + 1;
    }
  }
  __syncwarp();
  // ---- rank them: lanes 0..15 the first row's, 16..31 the second row's; with more than 16, each lane two
  const int h = lane >> 4, c = lane & 15;
  const int most = min(max(n[0], n[1]), kCandCap);
  const float* list = rs.cand_key[h];
  // Ranks below k that were found, 16 bits per row: their sum (at most 32 of at most 7) and how many above it.
  uint32_t found = 0;
  const float my0 = list[c];
  int r0 = 0;
  if (most <= 16) {
#pragma unroll 1
    for (int d = 0; d < most; d += 4) {
      const float4 o = *reinterpret_cast<const float4*>(list + d);
      count_greater(r0, o.x, my0); count_greater(r0, o.y, my0); count_greater(r0, o.z, my0); count_greater(r0, o.w, my0);
    }
  } else {
    const float my1 = list[c + 16];
    int r1 = 0;
#pragma unroll 1
    for (int d = 0; d < most; d += 4) {
      const float4 o = *reinterpret_cast<const float4*>(list + d);
      count_greater(r0, o.x, my0); count_greater(r0, o.y, my0); count_greater(r0, o.z, my0); count_greater(r0, o.w, my0);
      count_greater(r1, o.x, my1); count_greater(r1, o.y, my1); count_greater(r1, o.z, my1); count_greater(r1, o.w, my1);
    }
    if (my1 > -INFINITY && r1 < p.k) {
      rs.win[2 * pair + h][r1] = make_int2(__float_as_int(my1), rs.cand_id[h][c + 16]);
      found += 0x100u + r1;
    }
  }
  if (my0 > -INFINITY && r0 < p.k) {
    rs.win[2 * pair + h][r0] = make_int2(__float_as_int(my0), rs.cand_id[h][c]);
    found += 0x100u + r0;
  }
  // Anything but every rank found once means equal keys among the best (or too few candidates): such rows, and rows
  // whose list overflowed, take the plain path.  Equal keys share the first of their ranks: with k ranks found they
  // lower the sum, at the end of the list they raise the number found.  (A test for missing ranks alone would leave it
  // to the order of conflicting stores which of two equal keys at the last rank wins.)
  found = __reduce_add_sync(full, found << (16 * h));
  const uint32_t want = static_cast<uint32_t>(p.k) << 8 | static_cast<uint32_t>(p.k * (p.k - 1) / 2);
  if (found != (want | want << 16) || n[0] > kCandCap || n[1] > kCandCap) {
#pragma unroll 1
    for (int u = 0; u < 2; ++u) {
      if ((found >> (16 * u) & 0xffffu) == want && (u == 0 ? n[0] : n[1]) <= kCandCap) continue;
      // scratch: the row's staged words in this block, which nobody else reads (of a shared tile, a block
      // reads the other blocks' copies of its own slice only)
      float* keys = reinterpret_cast<float*>(__cvta_shared_to_generic(row_addr + u * stride));
      __syncwarp();
      for (int e = lane; e < p.E; e += 32) keys[e] = -INFINITY;
      __syncwarp();
#pragma unroll
      for (int j = 0; j < kCpl; ++j)
        if (j < lc.n && (u == 0 ? kept[0] : kept[1])) keys[lc.c0 + j] = u == 0 ? key[0][j] : key[1][j];
      __syncwarp();
      select_slow(keys, p.E, p.k, rs.win[2 * pair + u], lane);
    }
  }
}

// Expert ids, routing weights (Eq. 3's top-k with the model's weight rule) and histogram of up to 8 rows,
// four at a time: lane = (row, rank).
template <bool kSigmoid>
__device__ __forceinline__ void finish_rows(const RouterParams& p, RowsShared& sh, const RowScratch& rs, int n_rows,
                                            long long row0, int32_t* out_ids, float* out_w, int lane) {
  const uint32_t full = 0xffffffffu;
  const int rk = lane & 7;
  for (int base = 0; base < n_rows; base += 4) {
    const int i = base + (lane >> 3);
    const long long row = row0 + i;
    const bool valid = i < n_rows && row < p.T && rk < p.k;
    const int2 found = rs.win[i & 7][rk];
    const float key = __int_as_float(found.x);
    const int id = valid ? found.y : 0;
#ifdef FB_DEBUG
    // what the sanitizer would catch: a chosen expert outside [0, E), a repeated expert
    {
      bool bad = id < 0 || id >= p.E;
      for (int o = 1; o < 8; ++o) {
        const int other = __shfl_xor_sync(full, valid ? id : -1 - rk, o);
        bad = bad || (valid && other == id);
      }
      if (bad) atomicCAS(p.status, 0, FB_ERR_INTERNAL);
    }
#endif
    if (out_ids != nullptr && valid) out_ids[row * p.k + rk] = id;
    if (out_w != nullptr) {
      float w;
      if (kSigmoid) {
        w = valid ? key - sh.select_bias[id] : 0.0f;                        // unbiased sigmoid score
      } else {
        const float ref = __shfl_sync(full, key, lane & 24);                // row maximum of the keys
        w = valid ? __expf(key - ref) : 0.0f;
      }
      float sum = w;
      sum += __shfl_xor_sync(full, sum, 1);
      sum += __shfl_xor_sync(full, sum, 2);
      sum += __shfl_xor_sync(full, sum, 4);
      float scale;
      if (kSigmoid) scale = p.renorm ? p.route_scale / sum : p.route_scale;
      else scale = 1.0f / (p.renorm ? sum : rs.row_sum[i & 7]);
      if (valid) out_w[row * p.k + rk] = w * scale;
    }
    if (valid) atomicAdd(&sh.hist[id], 1u);
  }
}

// kCpl: columns per lane of the selection (gate_layout); kSigmoid: sigmoid + bias gate or softmax gate.
template <int kCpl, bool kSigmoid>
__global__ void __launch_bounds__(kRouterThreads, 1)
fb_router_rows_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_x2,
                      const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ RouterParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ RowsShared sh;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);      // warp-uniform for the compiler as well
  const int lane = threadIdx.x & 31;
  const uint32_t cluster_rank = cluster_ctarank();
  const uint32_t cta_rank = cluster_rank & 1u;               // which block of its pair
  const uint32_t lead_rank = cluster_rank & ~1u;             // the pair's even block
  const int J = p.pieces;
  const int piece = static_cast<int>(cluster_rank >> 1);
  const uint32_t stage_bytes = kATileBytes + static_cast<uint32_t>(p.N / 2) * kBlockK * 2;
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;   // swizzle atoms need 1024-byte alignment
  volatile int* abort_flag = &sh.abort_flag;
  FB_STAMP(0, 64);

  // Tile pairs of this cluster: pair_first, pair_first + pair_stride, ...  In kModeLayer the
  // first pairs_per_pass pairs belong to the early pass, the rest to the normal pass.
  const int pairs_per_pass = p.tiles_first / 2;
  const int total_pairs = p.mode == kModeLayer ? 2 * pairs_per_pass : pairs_per_pass;
  const int pair_first = static_cast<int>(blockIdx.x) / (2 * J);
  const int pair_stride = static_cast<int>(gridDim.x) / (2 * J);
  const bool several_tiles = pair_stride < total_pairs;
  // k-blocks of this pair
  const int kb0 = p.num_kb * piece / J, n_kb = p.num_kb * (piece + 1) / J - kb0;

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
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&sh.accum_bar[a]), static_cast<uint32_t>(p.issuers));   // one commit per MMA issuer
      mbar_init(smem_u32(&sh.tmem_empty_bar[a]), 2 * kEpilogueWarps);
    }
    mbar_init(smem_u32(&sh.staged_bar), static_cast<uint32_t>(J));
    fence_mbar_init();
    prefetch_tensormap(&tmap_x);
    if (p.mode == kModeLayer) prefetch_tensormap(&tmap_x2);
    prefetch_tensormap(&tmap_w);
  }
  if (warp == 1) {
    tmem_alloc<2>(smem_u32(&sh.tmem_base), static_cast<uint32_t>(p.tmem_cols));
    tmem_relinquish<2>();
  }
  if (warp >= 2) {
    const int et = threadIdx.x - 64;
    for (int e = et; e < FB_MAX_EXPERTS; e += kEpilogueThreads) sh.hist[e] = 0;
    if ((p.mode == kModePredictPlan || p.mode == kModeLayer) && !p.defer_counts) plan_clear(sh.plan, et, kEpilogueThreads);
  }
  tcgen05_fence_before();
  __syncthreads();
  cluster_arrive_relaxed(); cluster_wait();  // the other blocks' barriers and tensor memory are ready too
  tcgen05_fence_after();
  TileWalk walk;
  walk.pair_first = pair_first;
  walk.pair_stride = pair_stride;
  walk.total_pairs = total_pairs;
  walk.pairs_per_pass = pairs_per_pass;
  walk.kb0 = kb0;
  walk.n_kb = n_kb;
  walk.cluster_rank = cluster_rank;
  LoadPolicies policies = {0, 0};
  if (warp == 0) policies = load_policies(p);
  if (warp == kSecondIssuerWarp) prefetch_operands(p, &tmap_x, &tmap_x2, walk, &sh.started);
  // (see fb_router_kernel for these two)
  pdl_wait();
  if (threadIdx.x == 0) *static_cast<volatile int32_t*>(&sh.started) = 1;
  pdl_launch_dependents();
  const uint32_t tmem_base = sh.tmem_base;
  FB_STAMP(1, 64);
  bool closing_arrived = false;              // this warp has delivered its arrival for the closing cluster barrier

  if (warp == 0 || warp == 1 || warp == kSecondIssuerWarp) {
    if (warp == 0)
      produce_operands(p, &tmap_x, &tmap_x2, &tmap_w, walk, smem_base, stage_bytes, sh.full_bar, sh.empty_bar, policies, abort_flag);
    else if (cta_rank == 0 && (warp == 1 || p.issuers == 2))
      issue_mmas(p, walk, warp == 1 ? 0 : 1, tmem_base, smem_base, stage_bytes, sh.full_bar, sh.empty_bar, sh.accum_bar,
                 sh.tmem_empty_bar, sh.issuer_progress, abort_flag);
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue
    const int et = threadIdx.x - 64;                       // 0 .. kEpilogueThreads-1
    const int ew = warp - 2;
    const int quarter = warp & 3;                          // TMEM lanes this warp may touch
    const int sub = ew >> 2;                               // copies every fourth 16-column chunk
    const uint32_t taddr0 = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
    const uint32_t acc_sets = static_cast<uint32_t>(p.acc_sets), set_cols = static_cast<uint32_t>(p.issuers * p.N);
    const int E = p.E, N = p.N;
    const uint32_t row_stride = static_cast<uint32_t>(staging_stride(N)) * 4u;
    const bool two_acc = p.issuers == 2 && n_kb > 1;

    const LaneColumns lc = lane_columns(p, lane);
    // While the main loop runs, stage the biases and the placement for the planner (any block may
    // turn out to be the last one).
    for (int e = et; e < FB_MAX_EXPERTS; e += kEpilogueThreads) {
      sh.logit_bias[e] = (p.logit_bias != nullptr && e < E) ? p.logit_bias[e] : 0.0f;
      sh.select_bias[e] = (p.select_bias != nullptr && e < E) ? p.select_bias[e] : 0.0f;
    }
    for (int q = et; q < FB_MAX_EXPERTS / 4; q += kEpilogueThreads) sh.quad_word[q] = static_cast<uint16_t>(quad_word(p, q));
    float sb[kCpl];
#pragma unroll
    for (int j = 0; j < kCpl; ++j)
      sb[j] = (kSigmoid && p.select_bias != nullptr && j < lc.n) ? p.select_bias[lc.c0 + j] : 0.0f;
    if ((p.mode == kModePredictPlan || p.mode == kModeLayer) && !p.defer_counts) plan_load_placement(p.plan, sh.plan, et, kEpilogueThreads);

    uint32_t tiles_done = 0;
    uint32_t my_total = 0;                                   // expert et's assignments in this block's tiles for the index
    for (int pt = pair_first; pt < total_pairs; pt += pair_stride) {
      const bool second_pass = pt >= pairs_per_pass;
      const int mode = p.mode == kModeLayer ? (second_pass ? kModeDispatch : kModePredictPlan) : p.mode;
      const int tile = 2 * (second_pass ? pt - pairs_per_pass : pt) + static_cast<int>(cta_rank);
      // outputs of the normal pass are not written by tiles of the early pass
      int32_t* const out_ids = (p.mode == kModeLayer && !second_pass) ? p.early_ids : p.topk_ids;
      float* const out_logits = (p.mode == kModeLayer && !second_pass) ? p.early_logits : p.logits;
      float* const out_w = (p.mode == kModeLayer && !second_pass) ? nullptr : p.topk_w;
      const bool last_tile = pt + pair_stride >= total_pairs;

      // one thread polls for the finished accumulators, the others sleep at the barrier
      const uint32_t set = tiles_done % acc_sets, use = tiles_done / acc_sets;
      const uint32_t taddr = taddr0 + set * set_cols;
      if (et == 0) sh.accum_ok = mbar_wait<true>(smem_u32(&sh.accum_bar[set]), use & 1u, abort_flag) ? 1 : 0;
      named_bar_sync(kAccumBarrierId, kEpilogueThreads);
      bool got = sh.accum_ok != 0 && p.probe == 0;     // a measurement launch ends with its main loop
      if (sh.accum_ok == 0 && J == 1) break;                 // (blocks that share a tile pair go on and tell the others)
      ++tiles_done;
      tcgen05_fence_after();
      FB_STAMP(2, 64);

      // The last tile's staging reuses the operand ring, which is idle by then; earlier ones have
      // their own (smaller) area behind it and go through it a few rows at a time.
      const int chunk_rows = last_tile ? kTileM : p.chunk_rows;
      const uint32_t staging = smem_base + (last_tile ? 0u : static_cast<uint32_t>(p.stages) * stage_bytes);
      RowScratch& rs = reinterpret_cast<RowScratch*>(smem_raw + (staging - smem_u32(smem_raw)) +
                                                     static_cast<size_t>(chunk_rows) * row_stride)[ew];
      for (int r0 = 0; r0 < kTileM; r0 += chunk_rows) {
        if (r0 > 0) named_bar_sync(kPlanBarrierId, kEpilogueThreads);      // the previous rows have been read
        // ---- tensor memory -> shared memory: thread = row, 16 columns at a time
        if (quarter * 32 >= r0 && quarter * 32 < r0 + chunk_rows) {
          if (got) {
            const uint32_t dst = staging + static_cast<uint32_t>(quarter * 32 - r0 + lane) * row_stride;
#pragma unroll 1
            for (int c0 = sub * 16; c0 < N; c0 += kEpiSubs * 16) {
              uint32_t r[16], r2[16];
              tmem_ld_32x32b_x16(taddr + c0, r);
              if (two_acc) tmem_ld_32x32b_x16(taddr + N + c0, r2);
              tmem_ld_wait();
              if (two_acc) {                                 // add the odd k-blocks' accumulator
#pragma unroll
                for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(r2[j]));
              }
#pragma unroll
              for (int q = 0; q < 4; ++q)
                st_shared_v4(dst + static_cast<uint32_t>(sh.quad_word[c0 / 4 + q]) * 4u, r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
            }
          }
          tcgen05_fence_before();
          __syncwarp();
          // the issuers may overwrite the accumulators now
          if (several_tiles && lane == 0) mbar_arrive_cluster(smem_u32(&sh.tmem_empty_bar[set]), lead_rank);
        }
        FB_STAMP(3, 64);
        // ---- this warp's rows of the staged ones
        int first, count;
        if (J > 1) {
          // every block's partial tile is staged: one thread per block tells the others that share the tile (a
          // cluster barrier of all their warps took 0.9 us, every warp waiting for its own writes first)
          named_bar_sync(kPlanBarrierId, kEpilogueThreads);
          if (et < J) mbar_arrive_cluster(smem_u32(&sh.staged_bar), cta_rank + 2u * static_cast<uint32_t>(et));
          const bool staged = mbar_wait<true>(smem_u32(&sh.staged_bar), 0u, abort_flag);
          got = got && __all_sync(0xffffffffu, staged);
          const int slice = slice_rows(J), mine = min(slice, kTileM - piece * slice);
          const int per = (slice + 2 * kEpilogueWarps - 1) / (2 * kEpilogueWarps) * 2;
          first = piece * slice + ew * per;
          count = max(0, min(per, mine - ew * per));
        } else if (chunk_rows == kTileM) {
          // the four warps that share a quarter of the rows meet at their own barrier
          if (last_tile) {                                     // done with tensor memory and the partner
            // (releasing where arrivals at the partner's barriers may still be under way)
            if (several_tiles) cluster_arrive(); else cluster_arrive_relaxed();
            closing_arrived = true;
          }
          named_bar_sync(kRowBarrierBase + static_cast<uint32_t>(quarter), kEpiSubs * 32);
          first = quarter * 32 + sub * 8;
          count = 8;
        } else {
          named_bar_sync(kPlanBarrierId, kEpilogueThreads);
          const int per = chunk_rows / kEpilogueWarps;
          first = r0 + ew * per;
          count = per;
        }
        FB_STAMP(4, 64);
        const long long row0 = static_cast<long long>(tile) * kTileM + first;
        if (got && count > 0 && row0 < p.T) {
#pragma unroll 1
          for (int i = 0; i < count; i += 2)
            if (row0 + i < p.T)
              select_two_rows<kCpl, kSigmoid>(p, lc, sb, sh.logit_bias, staging + static_cast<uint32_t>(first - r0 + i) * row_stride,
                                              cluster_rank, row0 + i, out_logits, rs, i >> 1, lane);
          __syncwarp();
          FB_STAMP(8, 64);
          finish_rows<kSigmoid>(p, sh, rs, count, row0, out_ids, out_w, lane);
          FB_STAMP(10, 64);
        }
      }
      if (J > 1) { cluster_arrive_relaxed(); closing_arrived = true; }   // done with the other blocks' staged rows
      named_bar_sync(kPlanBarrierId, kEpilogueThreads);
      if (p.probe != 0) {
        // measurement launch: nothing is published
      } else if (mode == kModeDispatch || p.defer_counts) {
        const int slice = tile * J + piece;
        if (static_cast<long long>(tile) * kTileM + piece * slice_rows(J) < p.T) {  // (one beyond the last token owns no row)
          if (et < FB_MAX_EXPERTS) my_total += sh.hist[et];
          if (mode == kModeDispatch) write_slice_counts(p.slice_counts, slice, E, sh.hist, et);
        }
        if (last_tile) add_to_totals(mode == kModeDispatch ? p.totals : p.counts_scratch, E, my_total, et);
        if (several_tiles) {
          named_bar_sync(kPlanBarrierId, kEpilogueThreads);
          for (int e = et; e < E; e += kEpilogueThreads) sh.hist[e] = 0;
        }
      } else if (pt + pair_stride >= pairs_per_pass) {
        // The histogram keeps accumulating over this block's tiles of the pass and is published
        // once, after the last of them (one fence and one ticket per block, not per tile).
        publish_counts(sh, p, et, warp, lane, mode == kModePredictPlan && p.fuse_planner != 0);
      }
      FB_STAMP(12, 64);
    }
  }

  // ---------------------------------------------------------------- teardown
  // Tensor memory may be released, and a block may leave, only when all blocks of the cluster are
  // done with it: a warp delivers its arrival as soon as its own last access to the others is over, so
  // the wait normally finds the barrier complete.
  if (!closing_arrived) cluster_arrive();
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

}  // namespace fb
