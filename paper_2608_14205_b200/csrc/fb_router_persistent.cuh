// Persistent variant of the fused router kernel (Eqs. 2-5) for calls with more 128-row
// tiles than the GPU has SM pairs: every cluster of two blocks walks a strided list of
// tile pairs, and the epilogue of one tile runs while the tensor cores already work on the
// next one.
//
// What makes the overlap possible
//   * two accumulator sets alternate from tile to tile (256 columns fit twice since one issuer with one
//     accumulator keeps the tensor pipe busy at that width);
//   * the epilogue warps copy their share of the finished accumulators from tensor memory
//     into registers (64 columns per thread) and do all gating / selection work from registers;
//   * the epilogue's shared-memory scratch (group scores, candidate lists) has its own
//     44 KB behind the pipeline stages instead of reusing them.
// Restricted to the gates the ranking selection handles (DeepSeek-V3-like sigmoid gates with
// 32-expert groups, softmax gates over whole 32-column chunks); everything else, and
// every call that fits one tile per block, runs one of the other kernels.  Arithmetic, summation
// order and tie-breaking are those of fb_router_kernel, so both kernels give identical results.
//
// Warp roles as in fb_router_kernel.
#pragma once
#include "fb_router.cuh"

namespace fb {

constexpr int kPersistGroups = 8;            // 32-column chunks (= groups) per row, at most
constexpr size_t kPersistScratchBytes =
    (3 * kPersistGroups * kTileM + 2 * kCandCap * kTileM) * sizeof(float);   // 44 KB
static_assert(2 * kCandCap >= 2 * (kEpiSubs - 1) * FB_MAX_TOPK, "merge lists must fit in the candidate area");
static_assert(2 * kPersistGroups >= 2 * FB_MAX_TOPK, "result lists must fit in the group-score area");
static_assert(kPersistGroups == kBoundRows, "the three tables of best keys lie one after the other");

struct PersistShared {
  uint64_t full_bar[kMaxStages];
  uint64_t empty_bar[kMaxStages];
  // Two accumulator sets (of N columns per issuer) that alternate from tile to tile, so that the next
  // tile's MMAs need not wait for the drain.
  uint64_t accum_bar[2];                     // per set: both issuers' commits, once per use
  uint64_t tmem_empty_bar[2];                // per set, even block's copy: all epilogue warps of the pair, once per use
  uint64_t counts_bar;                       // odd block's copy: both blocks' early histograms are in counts_scratch
  uint32_t tmem_base;
  int32_t abort_flag;
  int32_t accum_ok;
  int32_t started;                           // the wait for the kernels before this one is over (prefetch_operands)
  int32_t tiles_done;                        // by this block, so far: restarts the limit of the wait on counts_bar
  int32_t any_unranked[4];                   // per row quarter: some row has too many or too few candidates
  int32_t issuer_progress[2];                // where both issuers use a stage: see issuer_turn_wait
  float logit_bias[FB_MAX_EXPERTS];
  alignas(16) float select_bias[FB_MAX_EXPERTS];
  alignas(16) uint32_t hist[FB_MAX_EXPERTS];          // early pass: over all of the block's tiles
  alignas(16) uint32_t tile_hist[2][FB_MAX_EXPERTS];  // normal pass: of one tile, in turn
  uint32_t cand_count[kTileM];
  PlanShared plan;
};

// End of the early pass, by the odd block's second issuer warp (idle there: the even block issues the pair's
// MMAs): once both blocks' histograms are in the scratch counts it takes the pair's ticket, and the last pair's
// publishes the count vector (Eq. 5), re-arms the scratch for the next call and runs the planner (Algorithm 1)
// when asked - beside the epilogue, which goes on with the next tile.  In the epilogue (publish_counts, as in the
// other router kernels) the planner held up its pair by 12 us and with it the end of the call: layer call with
// 131072 tokens, 128 experts 200.2 -> 198.2 us (226.2 -> 223.4 us in a loop).
__device__ __forceinline__ void finish_early_pass(PersistShared& sh, const RouterParams& p, int lane, volatile int* abort_flag) {
  const bool planner = p.mode != kModePredict && p.fuse_planner != 0;
  if (planner) {                                                    // any pair may turn out to be the last
    plan_clear(sh.plan, lane, 32);
    __syncwarp();
    plan_load_placement(p.plan, sh.plan, lane, 32);
    __syncwarp();
  }
  // (the end of a whole pass: under a pair limit a few pairs may walk millions of rows, so the limit is one tile's)
  if (!__all_sync(0xffffffffu, mbar_wait<true>(smem_u32(&sh.counts_bar), 0u, abort_flag, kWaitLimitNs, &sh.tiles_done))) return;
  int last = 0;
  if (lane == 0) {
    fence_acq_rel_gpu();                                            // what the two blocks added, before the ticket
    last = atomicAdd(p.ticket, 1u) == static_cast<uint32_t>(p.ticket_target) - 1 ? 1 : 0;
    if (last) fence_acq_rel_gpu();                                  // what the other pairs added
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return;
  for (int e = lane; e < p.E; e += 32) {
    const uint32_t c = __ldcg(&p.counts_scratch[e]);
    p.counts_out[e] = c;
    if (planner) plan_put_count(sh.plan, e, c);
    p.counts_scratch[e] = 0;                                        // ready for the next call
  }
  if (lane == 0) *p.ticket = 0;
  if (!planner) return;
  plan_swaps_apart(p.plan, sh.plan, lane, p.status, nullptr);
  __syncwarp();
  plan_write_placement(p.plan, sh.plan, lane, 32);
}

// kSigmoid: sigmoid + bias group-limited gate (true) or softmax gate (false); kLogitBias: a logit
// bias is given.  One instance per combination keeps code and registers to what it needs.
template <bool kSigmoid, bool kLogitBias>
__global__ void __launch_bounds__(kRouterThreads, 1)
fb_router_persistent_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_x2,
                            const __grid_constant__ CUtensorMap tmap_w, const __grid_constant__ RouterParams p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ PersistShared sh;

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);      // warp-uniform for the compiler as well
  const int lane = threadIdx.x & 31;
  const uint32_t cta_rank = cluster_ctarank();
  const uint32_t b_tile_bytes = static_cast<uint32_t>(p.N / 2) * kBlockK * 2;
  const uint32_t stage_bytes = kATileBytes + b_tile_bytes;
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  volatile int* abort_flag = &sh.abort_flag;

  // Tile pairs of this cluster: pair_first, pair_first + pair_stride, ...  In kModeLayer the
  // first pairs_per_pass pairs belong to the early pass, the rest to the normal pass.
  const int pairs_per_pass = p.tiles_first / 2;
  const int total_pairs = p.mode == kModeLayer ? 2 * pairs_per_pass : pairs_per_pass;
  const int pair_first = static_cast<int>(blockIdx.x) / 2;
  const int pair_stride = static_cast<int>(gridDim.x) / 2;

  if (threadIdx.x == 0) {
    sh.abort_flag = 0;
    sh.started = 0;
    sh.tiles_done = 0;
    for (int q = 0; q < 4; ++q) sh.any_unranked[q] = 0;
    sh.issuer_progress[0] = -1;
    sh.issuer_progress[1] = -1;
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(smem_u32(&sh.full_bar[s]), 1);
      mbar_init(smem_u32(&sh.empty_bar[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&sh.accum_bar[a]), static_cast<uint32_t>(p.issuers));
      mbar_init(smem_u32(&sh.tmem_empty_bar[a]), 2 * (kEpilogueThreads / 32));
    }
    mbar_init(smem_u32(&sh.counts_bar), 2);
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
    for (int e = et; e < FB_MAX_EXPERTS; e += kEpilogueThreads) {
      sh.hist[e] = 0;
      sh.tile_hist[0][e] = sh.tile_hist[1][e] = 0;
      if (e < kTileM) sh.cand_count[e] = 0;
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  cluster_arrive_relaxed(); cluster_wait();  // the partner's barriers and tensor memory are ready too
  tcgen05_fence_after();
  TileWalk walk;
  walk.pair_first = pair_first;
  walk.pair_stride = pair_stride;
  walk.total_pairs = total_pairs;
  walk.pairs_per_pass = pairs_per_pass;
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

  if (warp == kSecondIssuerWarp && cta_rank == 1) {
    if (p.mode != kModeDispatch && pair_first < pairs_per_pass) finish_early_pass(sh, p, lane, abort_flag);
  } else if (warp == 0 || warp == 1 || warp == kSecondIssuerWarp) {
    if (warp == 0)
      produce_operands(p, &tmap_x, &tmap_x2, &tmap_w, walk, smem_base, stage_bytes, sh.full_bar, sh.empty_bar, policies, abort_flag);
    else if (cta_rank == 0 && (warp == 1 || p.issuers == 2))
      issue_mmas(p, walk, warp == 1 ? 0 : 1, tmem_base, smem_base, stage_bytes, sh.full_bar, sh.empty_bar, sh.accum_bar,
                 sh.tmem_empty_bar, sh.issuer_progress, abort_flag);
  } else {
    // ------------------------------------------------------------ epilogue
    const int et = threadIdx.x - 64;                       // 0 .. kEpilogueThreads-1
    const int quarter = warp & 3;                          // TMEM lanes this warp may touch
    const int sub = (warp - 2) >> 2;                       // owns chunks sub and sub + 4
    const int row_in_tile = quarter * 32 + lane;
    const uint32_t taddr0 = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
    const uint32_t acc_sets = static_cast<uint32_t>(p.acc_sets), set_cols = static_cast<uint32_t>(p.issuers * p.N);
    const int E = p.E, N = p.N, k = p.k;
    constexpr bool sigmoid_gate = kSigmoid;
    const int n_chunks = E >> 5;                           // E is a multiple of 32 here
    constexpr bool has_lb = kLogitBias;
    const bool two_acc = p.issuers == 2 && p.num_kb > 1;
    // scratch behind the pipeline stages
    float* gscore_s = reinterpret_cast<float*>(smem_raw + (smem_base - smem_u32(smem_raw)) +
                                               static_cast<size_t>(p.stages) * stage_bytes);   // [8][128]
    float* glow_s = gscore_s + kPersistGroups * kTileM;                                         // [8][128]
    float* third_s = glow_s + kPersistGroups * kTileM;                                          // [8][128]
    // candidates [32][128]: ordered key bits in the high word, ~expert id in the low word
    unsigned long long* cand = reinterpret_cast<unsigned long long*>(third_s + kPersistGroups * kTileM);
    uint32_t* out_hi = reinterpret_cast<uint32_t*>(gscore_s);   // [8][128]: group scores are dead by then
    uint32_t* out_lo = reinterpret_cast<uint32_t*>(glow_s);

    // biases (read by these warps only, after the first barrier below)
    for (int e = et; e < FB_MAX_EXPERTS; e += kEpilogueThreads) {
      sh.logit_bias[e] = (p.logit_bias != nullptr && e < p.E) ? p.logit_bias[e] : 0.0f;
      sh.select_bias[e] = (p.select_bias != nullptr && e < p.E) ? p.select_bias[e] : 0.0f;
    }
    // Within a tile data passes only between the kEpiSubs warps that share a quarter of the rows: they meet at a
    // barrier of their own, and the histogram alternates between two tables, so that per tile two barriers of all
    // 16 warps are left (the accumulator's and the histogram's) of six.  131072 tokens, 128 experts: 203.0 -> 200.2 us
    // for the layer call; no difference at 16384 tokens, 256 experts.
    auto row_sync = [&]() { named_bar_sync(kRowBarrierBase + static_cast<uint32_t>(quarter), kEpiSubs * 32); };
    uint32_t tiles_done = 0;
    uint32_t my_total = 0;                                 // expert et's assignments in this block's tiles of the normal pass
    for (int pt = pair_first; pt < total_pairs; pt += pair_stride) {
      const bool second_pass = pt >= pairs_per_pass;
      const int mode = p.mode == kModeLayer ? (second_pass ? kModeDispatch : kModePredictPlan) : p.mode;
      const int tile = 2 * (second_pass ? pt - pairs_per_pass : pt) + static_cast<int>(cta_rank);
      const long long row = static_cast<long long>(tile) * kTileM + row_in_tile;
      const bool valid = row < p.T;
      int32_t* const out_ids = (p.mode == kModeLayer && !second_pass) ? p.early_ids : p.topk_ids;
      float* const out_w = (p.mode == kModeLayer && !second_pass) ? nullptr : p.topk_w;

      // one thread polls for the finished accumulators, the others sleep at the barrier
      const uint32_t set = tiles_done % acc_sets, use = tiles_done / acc_sets;
      const uint32_t taddr = taddr0 + set * set_cols;
      if (et == 0) sh.accum_ok = mbar_wait<true>(smem_u32(&sh.accum_bar[set]), use & 1u, abort_flag) ? 1 : 0;
      named_bar_sync(kAccumBarrierId, kEpilogueThreads);
      if (sh.accum_ok == 0) break;
      ++tiles_done;
      if (et == 0) *static_cast<volatile int32_t*>(&sh.tiles_done) = static_cast<int32_t>(tiles_done);
      tcgen05_fence_after();
      uint32_t* const hist = mode == kModeDispatch ? sh.tile_hist[tiles_done & 1u] : sh.hist;

      // ---------------- tensor memory -> registers: this thread's row, chunks sub and sub + 4
      float key[2][32];
#pragma unroll
      for (int ci = 0; ci < 2; ++ci) {
        const int c = sub + kEpiSubs * ci;
        if (c < n_chunks) {
          uint32_t r[32];
          tmem_ld_32x32b_x32(taddr + c * 32, r);
          tmem_ld_wait();
          if (two_acc) {                                     // add the odd k-blocks' accumulator
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              uint32_t r2[16];
              tmem_ld_32x32b_x16(taddr + N + c * 32 + 16 * h, r2);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 16; ++j)
                r[16 * h + j] = __float_as_uint(__uint_as_float(r[16 * h + j]) + __uint_as_float(r2[j]));
            }
          }
#pragma unroll
          for (int j = 0; j < 32; ++j) key[ci][j] = __uint_as_float(r[j]);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) key[ci][j] = -INFINITY;
        }
      }
      // the issuers may overwrite the accumulators now
      tcgen05_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(smem_u32(&sh.tmem_empty_bar[set]), 0u);

      // ---------------- selection keys in place; best two keys of every chunk
#pragma unroll
      for (int ci = 0; ci < 2; ++ci) {
        const int c = sub + kEpiSubs * ci;
        if (c < n_chunks) {
          const int c0 = c * 32;
          if (sigmoid_gate && !has_lb) {
            const float4* sb4 = reinterpret_cast<const float4*>(&sh.select_bias[c0]);
#pragma unroll
            for (int j4 = 0; j4 < 8; ++j4) {
              const float4 b = sb4[j4];
              key[ci][4 * j4 + 0] = fb_sigmoid(key[ci][4 * j4 + 0]) + b.x;
              key[ci][4 * j4 + 1] = fb_sigmoid(key[ci][4 * j4 + 1]) + b.y;
              key[ci][4 * j4 + 2] = fb_sigmoid(key[ci][4 * j4 + 2]) + b.z;
              key[ci][4 * j4 + 3] = fb_sigmoid(key[ci][4 * j4 + 3]) + b.w;
            }
          } else if (sigmoid_gate) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              key[ci][j] = fb_sigmoid(key[ci][j] + sh.logit_bias[c0 + j]) + sh.select_bias[c0 + j];
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) key[ci][j] = key[ci][j] + (has_lb ? sh.logit_bias[c0 + j] : 0.0f);
          }
          // four interleaved running (best, second, third) triples; the third only feeds the
          // softmax gate's bound
          float m1[4], m2[4], m3[4];
#pragma unroll
          for (int a = 0; a < 4; ++a) { m1[a] = -INFINITY; m2[a] = -INFINITY; m3[a] = -INFINITY; }
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float t = fminf(m1[j & 3], key[ci][j]);
            if (!sigmoid_gate) m3[j & 3] = fmaxf(m3[j & 3], fminf(m2[j & 3], t));
            m2[j & 3] = fmaxf(m2[j & 3], t);
            m1[j & 3] = fmaxf(m1[j & 3], key[ci][j]);
          }
#pragma unroll
          for (int a = 2; a >= 1; a >>= 1) {
#pragma unroll
            for (int b = 0; b < a; ++b) {
              // best three of two sorted triples
              const float lo1 = fminf(m1[b], m1[b + a]), hi2 = fmaxf(m2[b], m2[b + a]);
              if (!sigmoid_gate) m3[b] = fmaxf(fminf(lo1, hi2), fmaxf(m3[b], m3[b + a]));
              m2[b] = fmaxf(lo1, hi2);
              m1[b] = fmaxf(m1[b], m1[b + a]);
            }
          }
          glow_s[c * kTileM + row_in_tile] = m2[0];
          if (sigmoid_gate) {
            gscore_s[c * kTileM + row_in_tile] = group_score(m1[0], m2[0]);   // gs == 32
          } else {
            gscore_s[c * kTileM + row_in_tile] = m1[0];
            third_s[c * kTileM + row_in_tile] = m3[0];
          }
        }
      }
      row_sync();

      // ---------------- choose the groups; lower bound for the k-th key
      uint32_t kept = 0;
      float floor_key = INFINITY;
      if (sigmoid_gate) {
        float sc[kPersistGroups];
#pragma unroll
        for (int g = 0; g < kPersistGroups; ++g) sc[g] = g < n_chunks ? gscore_s[g * kTileM + row_in_tile] : -INFINITY;
#pragma unroll
        for (int g = 0; g < kPersistGroups; ++g) {
          int rank = 0;
#pragma unroll
          for (int h = 0; h < kPersistGroups; ++h)   // a lower-numbered group wins ties
            if (h != g) rank += (h < g ? sc[h] >= sc[g] : sc[h] > sc[g]) ? 1 : 0;
          if (g < n_chunks && rank < p.topk_group) {
            kept |= 1u << g;
            floor_key = fminf(floor_key, glow_s[g * kTileM + row_in_tile]);
          }
        }
      } else {
        // the k-th largest of the chunks' three best keys (3 n_chunks >= k of them)
        floor_key = kth_largest_known(gscore_s, n_chunks, k, row_in_tile);
        kept = (1u << n_chunks) - 1u;
      }
      // ---------------- collect the keys >= floor of this thread's kept chunks (the bound is one of
      // k known keys of the row, so at least k keys qualify; fewer only where keys are no numbers)
#pragma unroll
      for (int ci = 0; ci < 2; ++ci) {
        const int c = sub + kEpiSubs * ci;
        if (c < n_chunks && ((kept >> c) & 1u)) {
          uint32_t mine = 0;
#pragma unroll
          for (int j = 0; j < 32; ++j) mine += key[ci][j] >= floor_key ? 1u : 0u;
          const uint32_t first = atomicAdd(&sh.cand_count[row_in_tile], mine);
          // predicated stores, no branches: slot address advances past every hit, a hit is stored
          // while the slot is inside the list
          const uint32_t list = smem_u32(cand) + static_cast<uint32_t>(row_in_tile) * 8u;
          const uint32_t list_end = list + kCandCap * kTileM * 8u;
          uint32_t slot = list + first * (kTileM * 8u);
          const uint32_t id0 = ~static_cast<uint32_t>(c * 32);
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const uint32_t hit = key[ci][j] >= floor_key ? 1u : 0u;
            st_shared_v2_if(hit & (slot < list_end ? 1u : 0u), slot, id0 - j, ordered_bits(key[ci][j]));
            slot += hit * (kTileM * 8u);
          }
        }
      }
      row_sync();

      // ---------------- rank the candidates (many equal keys can overflow the list: handled below)
      const uint32_t n_cand = sh.cand_count[row_in_tile];
      if (n_cand < static_cast<uint32_t>(k)) sh.any_unranked[quarter] = 1;
      const bool overflow = rank_candidates(cand, n_cand, sub, row_in_tile, out_hi, out_lo);
      if (overflow) sh.any_unranked[quarter] = 1;
      row_sync();
      TopK top;
      top.init();
      if (sub == 0 && !overflow) read_ranked(top, k, out_hi, out_lo, row_in_tile);
      if (sh.any_unranked[quarter] != 0) {
        // Some of these rows had more than kCandCap keys at or above its floor (many equal
        // keys).  Such rows are selected by plain insertion: every thread scans its own kept
        // chunks in ascending expert order, then the row's first thread merges the lists.
        if (overflow) {
#pragma unroll
          for (int ci = 0; ci < 2; ++ci) {
            const int c = sub + kEpiSubs * ci;
            if (c < n_chunks && ((kept >> c) & 1u)) {
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (key[ci][j] > top.v[FB_MAX_TOPK - 1]) top.insert(key[ci][j], c * 32 + j);
            }
          }
          if (sub != 0) {
#pragma unroll
            for (int j = 0; j < FB_MAX_TOPK; ++j)            // the row's candidates are dead by now
              cand[((sub - 1) * FB_MAX_TOPK + j) * kTileM + row_in_tile] =
                  static_cast<unsigned long long>(__float_as_uint(top.v[j])) << 32 | static_cast<uint32_t>(top.i[j]);
          }
        }
        row_sync();
        if (overflow && sub == 0) {
#pragma unroll 1
          for (int j = 0; j < (kEpiSubs - 1) * FB_MAX_TOPK; ++j) {
            const unsigned long long w = cand[j * kTileM + row_in_tile];
            const float x = __uint_as_float(static_cast<uint32_t>(w >> 32));
            if (x > -INFINITY) top.insert_any_order(x, static_cast<int32_t>(static_cast<uint32_t>(w)));
          }
        }
        if (sub == 0) fill_missing_ranks(top, overflow ? ranks_taken(top) : sh.cand_count[row_in_tile], k);   // no numbers
      }

      if (sub == 0) sh.cand_count[row_in_tile] = 0;          // ready for the next tile

      // ---------------- outputs per row
      const bool writer = valid && sub == 0;
      if (writer) {
        // softmax gates reach this kernel only with renormalised weights: no denominator needed
        write_row_outputs(top, p, row, out_ids, out_w, sh.select_bias);
        // ---------------- histogram (Eq. 5)
#pragma unroll
        for (int j = 0; j < FB_MAX_TOPK; ++j)
          if (j < k) atomicAdd(&hist[top.i[j]], 1u);
      }
      named_bar_sync(kPlanBarrierId, kEpilogueThreads);
      if (et < 4) sh.any_unranked[et] = 0;                    // everyone has read it
      if (mode == kModeDispatch) {
        const bool owns = static_cast<long long>(tile) * kTileM < p.T;   // the padding block of an odd pair owns no tile
        if (owns) {
          if (et < FB_MAX_EXPERTS) my_total += hist[et];
          write_slice_counts(p.slice_counts, tile, E, hist, et);
        }
        if (pt + pair_stride >= total_pairs) add_to_totals(p.totals, E, my_total, et);
        // the other one was written out before the last barrier; the next tile counts into it
        for (int e = et; e < E; e += kEpilogueThreads) sh.tile_hist[(tiles_done & 1u) ^ 1u][e] = 0;
      } else if (pt + pair_stride >= pairs_per_pass) {
        // The histogram accumulated over this block's tiles of the pass and is handed on once, after the last of
        // them: the fence (cumulative over the barrier) and the arrival publish it to the pair's finishing warp.
        for (int e = et; e < E; e += kEpilogueThreads) {
          const uint32_t c = hist[e];
          if (c) atomicAdd(&p.counts_scratch[e], c);
        }
        named_bar_sync(kPlanBarrierId, kEpilogueThreads);
        if (et == 0) {
          fence_acq_rel_gpu();
          mbar_arrive_cluster(smem_u32(&sh.counts_bar), 1u);
        }
      }
    }
  }

  // ---------------------------------------------------------------- teardown
  tcgen05_fence_before();
  __syncthreads();
  cluster_arrive(); cluster_wait();          // nobody leaves while the partner may still signal it
  if (threadIdx.x == 0 && sh.abort_flag) atomicCAS(p.status, 0, FB_ERR_TIMEOUT);
  if (warp == 1) {
    tcgen05_fence_after();
    tmem_dealloc<2>(tmem_base, static_cast<uint32_t>(p.tmem_cols));
  }
}

}  // namespace fb
