// Host side of the C ABI declared in include/freebalance.h: argument checks, TMA
// descriptors, kernel launches.  No computation of the method happens on the host
// except the two pure helpers fb_budget_ns (Eq. 10) and fb_swap_cost_ns (Eq. 9).
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <mutex>
#include <new>

#include "../../include/freebalance.h"
#include "../../include/freebalance_aids.h"
#include "fb_dispatch.cuh"
#include "fb_migrate.cuh"
#include "fb_planner.cuh"
#include "fb_quality.cuh"
#include "fb_router.cuh"
#include "fb_router_persistent.cuh"
#include "fb_router_rows.cuh"

namespace {

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct MapEntry {
  const void* ptr = nullptr;
  int64_t rows = -1;
  uint32_t box_rows = 0;
  CUtensorMap map;
};

constexpr int kMapCache = 8;
constexpr size_t kLine = 32;            // words that blocks count on lie in lines of their own

// What a small kernel's launch asks of the SMs that its blocks go to: so much dynamic shared memory, and, where that is
// not zero, an execution priority.
struct SmShare {
  int smem = 0, priority = 0;
};
constexpr SmShare kAnyShare;

}  // namespace

struct fb_ctx {
  fb_config cfg;
  int device = 0;
  int N = 0;                      // experts padded to a multiple of 16 (UMMA N)
  fb::RouterParams gate;          // the shape- and gate-dependent fields of a launch (copied per call)
  bool ranking[2] = {false, false};    // the gate suits the ranking kernels [without / with routing weights]
  // One-tile ranking kernel: pipeline depth and dynamic shared memory
  int stages = 0;
  size_t smem_bytes = 0;
  // Persistent ranking kernel (several tiles per block pair)
  int persist_stages = 0;
  size_t persist_smem = 0;
  // Row-per-warp kernel: instance (log2 of the columns per lane), pipeline depth and dynamic shared memory
  // with one tile per block pair [0] and with several [1]
  int rows_kernel = 0;
  int rows_stages[2] = {0, 0};
  size_t rows_smem[2] = {0, 0};
  // [j]: clusters of 2 j blocks that fit on the GPU at once (j block pairs share a tile pair)
  int max_clusters[fb::kMaxPieces + 1] = {};
  int max_tiles = 0;
  int pair_limit = 0;             // the caller's limit on the block pairs to use (0 = none)
  int stage_limit = 0;            // diagnostic: pipeline stages at most (0 = as many as fit)
  int n_sm = 148;                 // SMs of the device
  SmShare own_sm;                 // for the planner kernel behind a router kernel (see launch_plan)
  int split_mode = 1;             // k-range split over the blocks of a cluster: 0 off, 1 on
  EncodeTiledFn encode = nullptr;
  // device scratch (one allocation from counts_scratch on but for slice_counts).  A prediction call may run beside a routing
  // call of the same context on another stream: they share no words of it.
  uint32_t* counts_scratch = nullptr;   // [256], zero between calls: the early pass's counts, prediction calls
  uint32_t* totals = nullptr;           // [256], zero between calls: sums of slice_counts
  uint32_t* layer_counts = nullptr;     // [256] directly behind them, zero between calls: the early pass's counts, layer calls
  uint32_t* ticket = nullptr;           // [2][kLine], zero between calls: prediction calls, layer calls
  uint32_t* index_ticket = nullptr;     // [1],   zero between calls
  int32_t* status = nullptr;            // [1]
  uint8_t* slice_counts = nullptr;      // [max_slices][slice_row_bytes(E)]: per-slice histograms for the dispatch index
  // descriptor cache
  MapEntry x_maps[kMapCache];
  MapEntry w_maps[kMapCache];
  int x_next = 0, w_next = 0;
  // staging for fb_layer_step_host (allocated on first use)
  bool staged = false;
  void* st_hprev = nullptr; void* st_H = nullptr;
  // staging for fb_apply_swaps_staged (allocated on first use): pinned host copy of a plan and of the
  // placement, and one device buffer of mig_stage_bytes
  void* mig_host = nullptr; void* mig_stage = nullptr; uint64_t mig_stage_bytes = 0;
  int32_t* st_pi = nullptr; int32_t* st_pi_out = nullptr;
  uint32_t* st_counts = nullptr; fb_swap* st_swaps = nullptr; int32_t* st_nswaps = nullptr;
  uint32_t* st_load_before = nullptr; uint32_t* st_load_after = nullptr;
  int32_t* st_ids = nullptr; float* st_w = nullptr;
  uint32_t* st_slot_offsets = nullptr; uint32_t* st_rank_offsets = nullptr;
  int32_t* st_perm = nullptr; int32_t* st_inv_perm = nullptr; uint32_t* st_rank_load = nullptr;
  uint64_t launches = 0;
  int fail_launch = 0;                                   // see fb_fail_launch
  uint64_t persistent_launches = 0;
  cudaEvent_t ev_before = nullptr, ev_after = nullptr;   // one-shot: recorded around the next router launch
  unsigned long long* stamps = nullptr;                  // caller's phase-stamp buffer (FB_TIMING builds)
  // attention profile (Eq. 10): one measurement per attention type, taken on the first layer of the type
  struct AttnSlot {
    int32_t layer = -1;                // r(l): the layer whose attention is (being) measured; -1 = none yet
    bool open = false;                 // begin recorded, end not yet
    bool pending = false;              // both events recorded, time not read yet
    bool has_time = false;
    uint64_t t_ns = 0;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
  } attn[FB_MAX_ATTENTION_TYPES];
};

namespace {

struct DeviceGuard {
  int prev = -1;
  bool ok = true;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) { ok = false; return; }
    if (prev != dev && cudaSetDevice(dev) != cudaSuccess) ok = false;
  }
  ~DeviceGuard() { if (prev >= 0) cudaSetDevice(prev); }
};

int next_pow2_at_least_32(int n) {
  int c = 32;
  while (c < n) c <<= 1;
  return c;
}

fb_status check_config(const fb_config& c) {
  if (c.T_max < 0 || c.d <= 0 || c.E <= 0 || c.k <= 0 || c.R <= 0) return FB_ERR_INVALID_ARG;
  if (c.gate != FB_GATE_SOFTMAX_TOPK && c.gate != FB_GATE_SIGMOID_GROUP_TOPK) return FB_ERR_INVALID_ARG;
  if (c.E > FB_MAX_EXPERTS || c.k > FB_MAX_TOPK || c.k > c.E) return FB_ERR_UNSUPPORTED_SHAPE;
  if (c.R > FB_MAX_RANKS || c.E % c.R != 0) return FB_ERR_UNSUPPORTED_SHAPE;
  if (c.d < 8 || c.d % 8 != 0) return FB_ERR_UNSUPPORTED_SHAPE;
  const int64_t widest = c.E > c.k ? c.E : c.k;
  if (static_cast<int64_t>(c.T_max) * widest >= (int64_t{1} << 31)) return FB_ERR_UNSUPPORTED_SHAPE;
  if (c.gate == FB_GATE_SIGMOID_GROUP_TOPK) {
    if (c.n_group <= 0 || c.topk_group <= 0) return FB_ERR_INVALID_ARG;
    if (c.n_group > FB_MAX_GROUPS || c.E % c.n_group != 0) return FB_ERR_UNSUPPORTED_SHAPE;
    if (c.topk_group > c.n_group || c.topk_group > FB_MAX_TOPK) return FB_ERR_UNSUPPORTED_SHAPE;
    if (static_cast<int64_t>(c.topk_group) * (c.E / c.n_group) < c.k) return FB_ERR_UNSUPPORTED_SHAPE;
  }
  return FB_OK;
}

fb_status make_map(fb_ctx* ctx, MapEntry* cache, int* next, const void* ptr, int64_t rows, uint32_t box_rows,
                   const CUtensorMap** out) {
  for (int i = 0; i < kMapCache; ++i)
    if (cache[i].ptr == ptr && cache[i].rows == rows && cache[i].box_rows == box_rows) {
      *out = &cache[i].map;
      return FB_OK;
    }
  if ((reinterpret_cast<uintptr_t>(ptr) & 15u) != 0) return FB_ERR_INVALID_ARG;
  MapEntry& e = cache[*next];
  *next = (*next + 1) % kMapCache;
  const cuuint64_t gdim[2] = {static_cast<cuuint64_t>(ctx->cfg.d), static_cast<cuuint64_t>(rows)};
  const cuuint64_t gstride[1] = {static_cast<cuuint64_t>(ctx->cfg.d) * 2};
  const cuuint32_t box[2] = {static_cast<cuuint32_t>(fb::kBlockK), box_rows};
  const cuuint32_t estride[2] = {1, 1};
  const CUresult r = ctx->encode(&e.map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), gdim, gstride,
                                 box, estride, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) { e.ptr = nullptr; e.rows = -1; return FB_ERR_CUDA; }
  e.ptr = ptr;
  e.rows = rows;
  e.box_rows = box_rows;
  *out = &e.map;
  return FB_OK;
}

uint64_t uniform_cost(const fb_budget& b, int cls) {
  const unsigned __int128 fs = static_cast<unsigned __int128>(b.expert_bytes) * 2u * b.fs_per_byte[cls];
  const unsigned __int128 ns = (fs + 999999u) / 1000000u + b.alpha_ns[cls];
  if (ns > UINT64_MAX) return 0;
  const uint64_t c = static_cast<uint64_t>(ns);
  return c < 1 ? 1 : c;
}

fb_status fill_plan(const fb_ctx* ctx, const fb_budget* b, const int32_t* pi, int32_t* pi_out, fb_swap* swaps,
                    int32_t* n_swaps, uint32_t* load_before, uint32_t* load_after, fb::PlanParams* pp) {
  if (!b || !pi || !pi_out || !n_swaps || !load_before || !load_after) return FB_ERR_INVALID_ARG;
  if (b->max_swaps > static_cast<uint32_t>(ctx->cfg.E / 2)) return FB_ERR_INVALID_ARG;
  if (b->max_swaps > 0 && !swaps) return FB_ERR_INVALID_ARG;
  if (b->gamma_num > FB_MAX_GAMMA_NUM) return FB_ERR_INVALID_ARG;
  pp->E = ctx->cfg.E;
  pp->R = ctx->cfg.R;
  pp->per_rank = pp->E / pp->R;
  pp->per_rank_inv = fb::per_rank_inverse(pp->per_rank);
  pp->max_swaps = b->max_swaps;
  pp->global_ns = b->global_ns;
  pp->rank_ns = b->rank_ns;
  pp->link_ns = b->link_ns;
  pp->tau_tokens = b->tau_tokens;
  pp->gamma_num = b->gamma_num;
  pp->gamma_den = b->gamma_den;
  for (int c = 0; c < 2; ++c) {
    pp->alpha_ns[c] = b->alpha_ns[c];
    pp->fs_per_byte[c] = b->fs_per_byte[c];
    pp->uniform_cost_ns[c] = uniform_cost(*b, c);
    if (b->expert_bytes_table == nullptr && pp->uniform_cost_ns[c] == 0) return FB_ERR_INVALID_ARG;
    pp->uniform_link_cap[c] = pp->uniform_cost_ns[c] ? b->link_ns / pp->uniform_cost_ns[c] : 0;
  }
  // Swaps the global budget carries when every swap costs the same, and whether the planner's uniform loop
  // has to keep books.  With one cost class a rank or a link is never charged more than the whole plan, so
  // a side budget that starts at or above the global one (the usual case: all three start at the same B) can
  // never stop a swap the global budget admits.
  pp->swap_cap = b->max_swaps;
  if (b->global_ns != FB_BUDGET_OFF && pp->uniform_cost_ns[0] != 0 && b->global_ns / pp->uniform_cost_ns[0] < pp->swap_cap)
    pp->swap_cap = static_cast<uint32_t>(b->global_ns / pp->uniform_cost_ns[0]);
  auto binds = [&](uint64_t side) { return side != FB_BUDGET_OFF && !(b->global_ns != FB_BUDGET_OFF && side >= b->global_ns); };
  const bool one_node = b->ranks_per_node <= 0 || b->ranks_per_node >= pp->R;
  pp->books = (!one_node || binds(b->rank_ns) || binds(b->link_ns)) ? 1 : 0;
  if (b->mode != FB_PLAN_LOOP && b->mode != FB_PLAN_SWEEP && b->mode != FB_PLAN_WIDE) return FB_ERR_INVALID_ARG;
  pp->mode = b->mode;
  pp->frontier_width = b->frontier_width;
  pp->ranks_per_node = b->ranks_per_node;
  pp->expert_bytes_table = b->expert_bytes_table;
  pp->expert_to_slot = pi;
  pp->expert_to_slot_out = pi_out;
  pp->swaps = swaps;
  pp->n_swaps = n_swaps;
  pp->load_before = load_before;
  pp->load_after = load_after;
  return FB_OK;
}

// Kernel instances of the ranking kernels by (gate, logit bias present), of the row-per-warp kernel by
// (log2 of the columns per lane, gate).
using RouterKernelFn = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, fb::RouterParams);
static RouterKernelFn ranking_kernel_fn(bool sigmoid, bool lb) {
  if (sigmoid) return lb ? fb::fb_router_kernel<true, true> : fb::fb_router_kernel<true, false>;
  return lb ? fb::fb_router_kernel<false, true> : fb::fb_router_kernel<false, false>;
}
static RouterKernelFn persistent_kernel_fn(bool sigmoid, bool lb) {
  if (sigmoid) return lb ? fb::fb_router_persistent_kernel<true, true> : fb::fb_router_persistent_kernel<true, false>;
  return lb ? fb::fb_router_persistent_kernel<false, true> : fb::fb_router_persistent_kernel<false, false>;
}
constexpr int kRowsKernels = 5;
static RouterKernelFn rows_kernel_fn(int log_cpl, bool sigmoid) {
  switch (2 * log_cpl + (sigmoid ? 1 : 0)) {
    case 0: return fb::fb_router_rows_kernel<1, false>;
    case 1: return fb::fb_router_rows_kernel<1, true>;
    case 2: return fb::fb_router_rows_kernel<2, false>;
    case 3: return fb::fb_router_rows_kernel<2, true>;
    case 4: return fb::fb_router_rows_kernel<4, false>;
    case 5: return fb::fb_router_rows_kernel<4, true>;
    case 6: return fb::fb_router_rows_kernel<8, false>;
    case 7: return fb::fb_router_rows_kernel<8, true>;
    case 8: return fb::fb_router_rows_kernel<16, false>;
    default: return fb::fb_router_rows_kernel<16, true>;
  }
}

// Launch of a small kernel that may start under the end of the stream's previous kernel (it waits for
// that kernel's completion - griddepcontrol.wait - before it touches global memory).
template <typename... Params, typename... Args>
cudaError_t launch_dependent(void (*kernel)(Params...), int blocks, int threads, const SmShare& share, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(static_cast<unsigned>(blocks), 1, 1);
  cfg.blockDim = dim3(static_cast<unsigned>(threads), 1, 1);
  cfg.dynamicSmemBytes = static_cast<size_t>(share.smem);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributePriority;
  attr[1].val.priority = share.priority;
  cfg.attrs = attr;
  cfg.numAttrs = share.smem > 0 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// One of a context's launches: counted, and with fb_fail_launch one of them is not made.
bool launch_refused(fb_ctx* ctx) {
  ++ctx->launches;
  return ctx->fail_launch > 0 && --ctx->fail_launch == 0;
}
template <typename... Params, typename... Args>
cudaError_t launch_counted(fb_ctx* ctx, void (*kernel)(Params...), int blocks, int threads, const SmShare& share, cudaStream_t stream, Args... args) {
  return launch_refused(ctx) ? cudaErrorUnknown : launch_dependent(kernel, blocks, threads, share, stream, args...);
}

// A kernel that should have read and cleared these of the context's words was not launched behind the router kernel that
// adds to them: back to zero for the next call.
void clear_unread(uint32_t* words, int sets, cudaStream_t stream) {
  cudaMemsetAsync(words, 0, static_cast<size_t>(sets) * FB_MAX_EXPERTS * sizeof(uint32_t), stream);
}

// counts_out: counts are the totals of a prediction pass (see fb_plan_kernel).
// share: behind a router kernel the block asks for an SM of its own (all of the shared memory), ahead of other kernels' blocks
// (the highest priority).  It is launched while the router blocks run, and beside another stream's kernel - the attention that
// the prediction is meant to run beside - the only SMs with room for it would be the busy ones of that kernel, where its one
// deciding warp starved; without the priority the SM that the first router block leaves went to that kernel's waiting blocks.
// Prediction and plan of 8192 x 128 beside a kernel of multiply-adds: on 32 pairs, the other SMs taken, 99 us without either
// and 24 with; on all SMs, with the other kernel launched 2 us later, 109 without either, 611 with the SM alone, 23 with both.
fb_status launch_plan(fb_ctx* ctx, const fb::PlanParams& pp, uint32_t* counts, uint32_t* counts_out, const SmShare& share,
                      cudaStream_t stream) {
  const cudaError_t err = launch_counted(ctx, fb::plan_needs_general_loop(pp) ? fb::fb_plan_kernel<true> : fb::fb_plan_kernel<false>,
                                         1, fb::kPlanThreads, share, stream, pp, counts, counts_out, ctx->status);
  return err == cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

// Launch a router kernel in one of its modes.
// x2 is the second input of kModeLayer (the normal router input), nullptr otherwise.
// *pieces_out (optional): block pairs per tile pair, i.e. row slices per tile of the histogram table.
// *deferred_out (layer calls): the dispatch-index kernel has to count and plan.
fb_status launch_router(fb_ctx* ctx, const fb_router* router, const void* x, int32_t T, int mode,
                        uint32_t* counts_out, int32_t* topk_ids, float* topk_w, float* logits,
                        const fb::PlanParams* plan, cudaStream_t stream, const void* x2 = nullptr, int probe = 0,
                        int* pieces_out = nullptr, bool* deferred_out = nullptr, int32_t* early_ids = nullptr,
                        float* early_logits = nullptr) {
  const CUtensorMap *mx = nullptr, *mx2 = nullptr, *mw = nullptr;
  fb_status st = make_map(ctx, ctx->x_maps, &ctx->x_next, x, T, fb::kTileM, &mx);
  if (st != FB_OK) return st;
  const CUtensorMap map_x = *mx;     // by value: the second lookup may evict the cache slot mx points to
  mx = &map_x;
  mx2 = mx;
  if (mode == fb::kModeLayer) {
    st = make_map(ctx, ctx->x_maps, &ctx->x_next, x2, T, fb::kTileM, &mx2);
    if (st != FB_OK) return st;
  }
  st = make_map(ctx, ctx->w_maps, &ctx->w_next, router->W, ctx->cfg.E, static_cast<uint32_t>(ctx->N / 2), &mw);
  if (st != FB_OK) return st;
  const fb_config& c = ctx->cfg;
  fb::RouterParams p = ctx->gate;
  p.T = T;
  p.mode = mode;
  p.logit_bias = router->logit_bias;
  p.select_bias = c.gate == FB_GATE_SIGMOID_GROUP_TOPK ? router->select_bias : nullptr;
  const bool layer = mode == fb::kModeLayer;
  p.counts_scratch = layer ? ctx->layer_counts : ctx->counts_scratch;
  p.ticket = ctx->ticket + (layer ? kLine : 0);
  p.status = ctx->status;
  p.counts_out = counts_out;
  p.topk_ids = topk_ids;
  p.topk_w = topk_w;
  p.logits = logits;
  p.early_ids = early_ids;
  p.early_logits = early_logits;
  p.slice_counts = ctx->slice_counts;
  p.totals = ctx->totals;
  p.stamps = ctx->stamps;
  p.probe = probe;
  if (plan) p.plan = *plan;
  // A launch of more tiles than the GPU holds at once plans itself (fuse_planner); a plan that needs the general loop (per-expert sizes, a
  // planner variant) gets the planner kernel behind the router kernel instead.
  const bool plan_wanted = plan != nullptr && (mode == fb::kModePredictPlan || mode == fb::kModeLayer);
  p.fuse_planner = (plan_wanted && !fb::plan_needs_general_loop(*plan)) ? 1 : 0;
  const int tiles = (T + fb::kTileM - 1) / fb::kTileM;
  p.tiles_first = (tiles + 1) / 2 * 2;                            // a pair never straddles the two passes
  const int tile_pairs = (mode == fb::kModeLayer ? 2 : 1) * (p.tiles_first / 2);
  const int pairs_avail = ctx->pair_limit > 0 && ctx->pair_limit < ctx->max_clusters[1] && probe == 0
                              ? ctx->pair_limit : ctx->max_clusters[1];
  // Few tile pairs: as many block pairs per tile pair as fit at once (all clusters of the launch
  // are resident together) and have at least two k-blocks each.  Numbers that are not powers of two only
  // where they shorten a pair's piece by three k-blocks or more: prediction and plan of 4300 x 7168 with 256 experts
  // takes 37.7 us with two pairs and 31.9 with three, of 2048 x 4096 with 8 experts 12.41 with four (16 k-blocks
  // each) and 12.03 with five (13); but a layer call of 900 x 2048 with 128 experts 19.85 with four (8 k-blocks
  // each) and 20.02 with five (7).
  int J = 1, power = 1;
  if (ctx->split_mode != 0 && probe == 0)
    for (int j = 2; j <= fb::kMaxPieces; ++j) {
      if (tile_pairs > ctx->max_clusters[j] || tile_pairs * j > pairs_avail || p.num_kb < 2 * j) continue;
      if ((j & (j - 1)) == 0) J = power = j;
      else if ((p.num_kb + power - 1) / power - (p.num_kb + j - 1) / j >= 3) J = j;
    }
  p.pieces = J;
  if (pieces_out) *pieces_out = J;
  // Which kernel: whole tiles of a gate that the ranking selection handles go there (one tile per pair,
  // or several where more tile pairs than block pairs fit or than the caller allows); tiles shared by
  // several pairs and all other gates take the row-per-warp selection (figures: fb_router_rows.cuh).
  // Logit dumps: a block of the ranking kernel writes its rows from registers, 16 bytes a store (row-per-warp selection for
  // dumps instead: serving step with 8192 tokens, 128 experts 75.4 us against 71.6), one tile per pair.  A dump that does
  // not start on 16 bytes goes to the row-per-warp selection, which stores single words, and so does one whose caller
  // limits the pairs: that kernel writes logits while it walks several tiles.
  const bool dump = logits != nullptr || early_logits != nullptr;
  const bool over_limit = pairs_avail < ctx->max_clusters[1] && tile_pairs > pairs_avail;
  const bool whole_vectors = (reinterpret_cast<uintptr_t>(logits) | reinterpret_cast<uintptr_t>(early_logits)) % 16 == 0;
  const bool ranking = J == 1 && ctx->ranking[topk_w != nullptr ? 1 : 0] && whole_vectors && !(dump && over_limit);
  const bool several = J == 1 && probe == 0 && tile_pairs > pairs_avail && !(ranking && dump);
  // Both passes of the layer at the same time: nothing could hide the planner behind the second pass, so
  // the dispatch-index kernel counts and plans (see fb_dispatch_kernel).  With several tiles per pair the
  // early pass is done long before the normal one and the planner runs beside it.
  const bool tile_per_block = (T + fb::kDispatchTile - 1) / fb::kDispatchTile <= ctx->n_sm;   // of that kernel
  // A prediction pass that plans hands its counts to the planner kernel where one tile per pair leaves nothing to hide it behind.
  const bool layer_plan = mode == fb::kModeLayer && tile_per_block && p.fuse_planner && deferred_out != nullptr;
  const bool pass_plan = mode == fb::kModePredictPlan && plan_wanted;
  p.defer_counts = (!several && probe == 0 && (layer_plan || pass_plan)) ? 1 : 0;
  if (p.defer_counts) {
    p.fuse_planner = 0;
    if (deferred_out != nullptr) *deferred_out = true;
  }
  int clusters = tile_pairs;
  if (several) {
    // no more pairs than the number of rounds needs: 128 tile pairs run as 2 rounds on 64
    // block pairs just as fast as on 74 (measured), and the other SMs stay free for other streams
    const int rounds = (tile_pairs + pairs_avail - 1) / pairs_avail;
    clusters = (tile_pairs + rounds - 1) / rounds;
    // two accumulator sets: 512 tensor-memory columns at most
    p.acc_sets = 2;
    p.tmem_cols = next_pow2_at_least_32(2 * p.issuers * ctx->N);
  }
  const int blocks = 2 * J * clusters;
  p.prefetch_kb = probe == 0 ? fb::kPrefetchBytes / fb::kATileBytes / blocks : 0;
  // every block publishes its counts once: as many tickets as blocks that own a tile of the counted pass
  p.ticket_target = blocks < p.tiles_first * J ? blocks : p.tiles_first * J;
  RouterKernelFn fn;
  size_t smem;
  const bool sigmoid = c.gate == FB_GATE_SIGMOID_GROUP_TOPK;
  if (!ranking) {
    fn = rows_kernel_fn(ctx->rows_kernel, sigmoid);
    p.stages = ctx->rows_stages[several ? 1 : 0];
    smem = ctx->rows_smem[several ? 1 : 0];
  } else if (several) {
    fn = persistent_kernel_fn(sigmoid, router->logit_bias != nullptr);
    p.ticket_target /= 2;                      // one ticket per pair there
    p.stages = ctx->persist_stages;
    smem = ctx->persist_smem;
  } else {
    fn = ranking_kernel_fn(sigmoid, router->logit_bias != nullptr);
    p.stages = ctx->stages;
    smem = ctx->smem_bytes;
  }
  if (ctx->stage_limit >= 2 && ctx->stage_limit < p.stages) p.stages = ctx->stage_limit;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(static_cast<unsigned>(blocks), 1, 1);
  cfg.blockDim = dim3(fb::kRouterThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  if (ctx->ev_before) cudaEventRecord(ctx->ev_before, stream);
  // Programmatic dependent launch: this kernel's set-up overlaps the previous kernel's execution (where
  // that one allows it, as the library's kernels do); the kernel waits for its completion
  // (griddepcontrol.wait) before it reads any global memory.
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned>(2 * J);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  const cudaError_t err = launch_refused(ctx) ? cudaErrorUnknown : cudaLaunchKernelEx(&cfg, fn, *mx, *mx2, *mw, p);
  if (ctx->ev_after) cudaEventRecord(ctx->ev_after, stream);
  ctx->ev_before = ctx->ev_after = nullptr;
  if (several) ++ctx->persistent_launches;
  if (err != cudaSuccess) return FB_ERR_CUDA;
  if (pass_plan && p.defer_counts) {
    st = launch_plan(ctx, *plan, p.counts_scratch, counts_out, ctx->own_sm, stream);
    if (st != FB_OK) clear_unread(p.counts_scratch, 1, stream);
  } else if (plan_wanted && !p.fuse_planner && !p.defer_counts) {
    st = launch_plan(ctx, *plan, counts_out, nullptr, ctx->own_sm, stream);
    if (st != FB_OK && layer) clear_unread(ctx->totals, 1, stream);     // no dispatch index follows
  }
  return st;
}

// Dispatch index from the router kernel's top-k ids and per-slice histograms.  plan: also the count vector and
// the plan, from the early pass's histograms (one tile per block only; expert_to_slot is then the placement
// before the plan, and the index is made under the one after it).
fb_status launch_dispatch_index(fb_ctx* ctx, int32_t T, int slices_per_tile, const fb::PlanParams* plan,
                                uint32_t* counts_out, const int32_t* expert_to_slot, const int32_t* topk_ids,
                                uint32_t* slot_offsets, uint32_t* rank_offsets, int32_t* perm, int32_t* inv_perm,
                                uint32_t* rank_load, cudaStream_t stream) {
  const fb_config& c = ctx->cfg;
  fb::DispatchParams dp;
  memset(&dp, 0, sizeof(dp));
  dp.T = T; dp.k = c.k; dp.E = c.E; dp.R = c.R; dp.per_rank = c.E / c.R;
  dp.num_tiles = (T + fb::kDispatchTile - 1) / fb::kDispatchTile;
  dp.topk_ids = topk_ids;
  dp.slices_per_tile = slices_per_tile;
  const int rows = fb::slice_rows(slices_per_tile);
  dp.num_slices = T / fb::kDispatchTile * slices_per_tile + (T % fb::kDispatchTile + rows - 1) / rows;
  dp.slice_counts = ctx->slice_counts;
  dp.totals = ctx->totals;
  dp.ticket = ctx->index_ticket;
  dp.counts_out = counts_out;
  if (plan) dp.plan = *plan;
  dp.expert_to_slot = expert_to_slot;
  dp.slot_offsets = slot_offsets;
  dp.rank_offsets = rank_offsets;
  dp.perm = perm;
  dp.inv_perm = inv_perm;
  dp.rank_load = rank_load;
  dp.status = ctx->status;
  dp.stamps = ctx->stamps;
  // one block per SM at most: more tiles than that are walked in runs (every block reads up to half of the
  // histogram table, so more blocks would only read it more often)
  const int blocks = dp.num_tiles < ctx->n_sm ? dp.num_tiles : ctx->n_sm;
  const cudaError_t err = launch_counted(ctx, blocks < dp.num_tiles ? fb::fb_dispatch_runs_kernel
                                              : plan != nullptr     ? fb::fb_dispatch_kernel<true>
                                                                    : fb::fb_dispatch_kernel<false>,
                                         blocks, fb::kDispatchThreads, kAnyShare, stream, dp);
  if (err == cudaSuccess) return FB_OK;
  clear_unread(ctx->totals, plan != nullptr ? 2 : 1, stream);
  return FB_ERR_CUDA;
}

// The device that owns a device pointer (-1 if it is not device memory).
int device_of(const void* p) {
  cudaPointerAttributes pa;
  if (cudaPointerGetAttributes(&pa, p) != cudaSuccess) { cudaGetLastError(); return -1; }
  return (pa.type == cudaMemoryTypeDevice || pa.type == cudaMemoryTypeManaged) ? pa.device : -1;
}

// A fixed one-swap plan over two slots for fb_calibrate_exchange: [placement: 2][swap: 4][n: 1].
// Constant data inside the library image, so the calibration allocates nothing.
__device__ const int32_t g_calibration_plan[8] = {0, 1, 0, 1, 0, 1, 1, 0};

template <typename Tp>
bool dev_alloc(Tp** p, size_t count) {
  return cudaMalloc(reinterpret_cast<void**>(p), (count ? count : 1) * sizeof(Tp)) == cudaSuccess;
}

}  // namespace

// What the host side needs to know of a device.  Three attributes: the whole property record takes the driver 2.5 ms
// and, with other processes on the machine, now and then a hundred (2.9 -> 0.4 ms per context).
struct DeviceLimits {
  int n_sm = 0, smem_optin = 0;
  bool usable = false;                                 // built for sm_100a only; no fallback
};
static DeviceLimits device_limits(int device) {
  DeviceLimits d;
  int major = 0;
  d.usable = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device) == cudaSuccess && major == 10 &&
             cudaDeviceGetAttribute(&d.n_sm, cudaDevAttrMultiProcessorCount, device) == cudaSuccess &&
             cudaDeviceGetAttribute(&d.smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device) == cudaSuccess;
  return d;
}

// Shape-dependent launch parameters of the router kernels (host arithmetic only): padded width, TMEM
// columns, gate layout, pipeline depths and dynamic shared memory.
static fb_status setup_router_shape(fb_ctx* ctx, const DeviceLimits& dev) {
  const fb_config& c = ctx->cfg;
  ctx->N = (c.E + 15) / 16 * 16;
  fb::RouterParams& g = ctx->gate;
  memset(&g, 0, sizeof(g));
  g.d = c.d; g.E = c.E; g.N = ctx->N; g.k = c.k;
  g.gate = c.gate;
  g.n_group = c.gate == FB_GATE_SIGMOID_GROUP_TOPK ? c.n_group : 1;
  g.topk_group = c.gate == FB_GATE_SIGMOID_GROUP_TOPK ? c.topk_group : 1;
  g.renorm = c.renorm; g.route_scale = c.route_scale;
  g.num_kb = (c.d + fb::kBlockK - 1) / fb::kBlockK;
  g.issuers = ctx->N <= 128 ? 2 : 1;                             // the reason is in fb_router.cuh
  g.acc_sets = 1;
  g.tmem_cols = next_pow2_at_least_32(g.issuers * ctx->N);
  const int cpl = fb::gate_layout(c.E, c.gate, c.n_group, c.topk_group, &g);
  ctx->rows_kernel = 0;
  while ((1 << ctx->rows_kernel) < cpl) ++ctx->rows_kernel;
  if (ctx->rows_kernel >= kRowsKernels) return FB_ERR_UNSUPPORTED_SHAPE;   // (no gate within the limits has more columns per lane)
  const size_t optin = static_cast<size_t>(dev.smem_optin) - 2048 - 1024;
  const size_t stage_bytes = fb::kATileBytes + static_cast<size_t>(ctx->N / 2) * fb::kBlockK * 2;
  auto depth = [&](size_t bytes) {
    const int n = static_cast<int>(bytes / stage_bytes);
    return n > fb::kMaxStages ? fb::kMaxStages : n;
  };
  for (int w = 0; w < 2; ++w)
    ctx->ranking[w] = fb::ranking_gate(c.E, c.k, c.gate, g.n_group, g.topk_group,
                                       w != 0 && !c.renorm && c.gate == FB_GATE_SOFTMAX_TOPK);
  if (ctx->ranking[0]) {
    size_t budget = optin - sizeof(fb::RouterShared);
    ctx->stages = depth(budget);
    size_t dyn = ctx->stages * stage_bytes;
    if (dyn < fb::epilogue_scratch_bytes(ctx->N)) dyn = fb::epilogue_scratch_bytes(ctx->N);
    ctx->smem_bytes = dyn + 1024;
    if (ctx->stages < 2 || dyn > budget) return FB_ERR_UNSUPPORTED_SHAPE;
    budget = optin - sizeof(fb::PersistShared);
    ctx->persist_stages = depth(budget - fb::kPersistScratchBytes);
    ctx->persist_smem = ctx->persist_stages * stage_bytes + fb::kPersistScratchBytes + 1024;
    if (ctx->persist_stages < 2) return FB_ERR_UNSUPPORTED_SHAPE;
  }
  // one tile per pair: the staged logits reuse the ring
  const size_t budget = optin - sizeof(fb::RowsShared);
  const size_t full_staging = fb::staging_bytes(fb::kTileM, ctx->N);
  ctx->rows_stages[0] = depth(budget);
  size_t dyn = ctx->rows_stages[0] * stage_bytes;
  if (dyn < full_staging) dyn = full_staging;
  if (ctx->rows_stages[0] < 2 || dyn > budget) return FB_ERR_UNSUPPORTED_SHAPE;
  ctx->rows_smem[0] = dyn + 1024;
  // several tiles per pair: staging of its own behind the ring, as many rows at a time as leave five
  // stages (128 rows of up to 144 columns, 32 rows of 256)
  for (int rows = fb::kTileM; rows >= 32; rows /= 2) {
    const size_t staging = fb::staging_bytes(rows, ctx->N);
    ctx->rows_stages[1] = depth(budget - staging);
    dyn = ctx->rows_stages[1] * stage_bytes + staging;
    if (dyn < full_staging) dyn = full_staging;                  // the last tile stages all rows over the ring
    ctx->rows_smem[1] = dyn + 1024;
    g.chunk_rows = rows;
    if (ctx->rows_stages[1] >= 5) break;
  }
  if (ctx->rows_stages[1] < 2) return FB_ERR_UNSUPPORTED_SHAPE;
  ctx->max_tiles = (c.T_max + fb::kTileM - 1) / fb::kTileM;
  ctx->n_sm = dev.n_sm;
  return FB_OK;
}

// What is set or asked once per device, for all contexts:
//   * The ceiling on a kernel's dynamic shared memory belongs to the function on a device, not to a context: contexts of
//     different shapes share the kernel instances.  It is raised for every router kernel instance to the most the
//     device allows beside the kernel's static shared memory, and never lowered again (so for the planner kernel).
//   * How many clusters of 2, 4, .. 16 blocks the GPU holds at once.  Every router launch takes more than half of an
//     SM's shared memory (the operand ring alone is 136 KB or more at any width), so one block fits an SM and the answer
//     is the same for all instances and shapes.
static fb_status set_up_device(fb_ctx* ctx, int device, const DeviceLimits& dev) {
  static std::mutex mutex;
  static struct { bool ready; int max_clusters[fb::kMaxPieces + 1]; SmShare own_sm; } known[64] = {};
  std::lock_guard<std::mutex> lock(mutex);
  if (device >= 0 && device < 64 && known[device].ready) {
    memcpy(ctx->max_clusters, known[device].max_clusters, sizeof(ctx->max_clusters));
    ctx->own_sm = known[device].own_sm;
    return FB_OK;
  }
  bool ok = true;
  auto raise = [&](const void* fn) -> int {
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess) { ok = false; return 0; }
    const int most = dev.smem_optin - static_cast<int>(fa.sharedSizeBytes);
    ok = ok && most > 0 && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, most) == cudaSuccess;
    return most;
  };
  auto raise_router = [&](RouterKernelFn fn_) -> int {
    const void* fn = reinterpret_cast<const void*>(fn_);
    const int most = raise(fn);
    ok = ok && cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;   // clusters of 16
    return most;
  };
  for (int i = 0; i < 4; ++i) {
    raise_router(ranking_kernel_fn(i / 2 != 0, i % 2 != 0));
    raise_router(persistent_kernel_fn(i / 2 != 0, i % 2 != 0));
  }
  int smem = 0;
  for (int i = 0; i < 2 * kRowsKernels; ++i) smem = raise_router(rows_kernel_fn(i / 2, i % 2 != 0));
  const int plan_general = raise(reinterpret_cast<const void*>(fb::fb_plan_kernel<true>));
  const int plan_uniform = raise(reinterpret_cast<const void*>(fb::fb_plan_kernel<false>));
  ctx->own_sm.smem = plan_general < plan_uniform ? plan_general : plan_uniform;
  int least = 0;
  ok = ok && cudaDeviceGetStreamPriorityRange(&least, &ctx->own_sm.priority) == cudaSuccess;
  if (!ok) { cudaGetLastError(); return FB_ERR_CUDA; }
  cudaLaunchConfig_t occ;
  memset(&occ, 0, sizeof(occ));
  occ.blockDim = dim3(fb::kRouterThreads, 1, 1);
  occ.dynamicSmemBytes = static_cast<size_t>(smem);
  cudaLaunchAttribute cl[1];
  cl[0].id = cudaLaunchAttributeClusterDimension;
  occ.attrs = cl;
  occ.numAttrs = 1;
  for (int j = 1; j <= fb::kMaxPieces; ++j) {
    cl[0].val.clusterDim.x = 2u * j; cl[0].val.clusterDim.y = 1; cl[0].val.clusterDim.z = 1;
    occ.gridDim = dim3(2u * j * static_cast<unsigned>(dev.n_sm), 1, 1);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, rows_kernel_fn(kRowsKernels - 1, true), &occ) != cudaSuccess) n = 0;
    ctx->max_clusters[j] = n;
  }
  cudaGetLastError();
  if (ctx->max_clusters[1] < 1) return FB_ERR_CUDA;
  if (device >= 0 && device < 64) {
    memcpy(known[device].max_clusters, ctx->max_clusters, sizeof(ctx->max_clusters));
    known[device].own_sm = ctx->own_sm;
    known[device].ready = true;
  }
  return FB_OK;
}

// Rows of the histogram table: a launch that cuts its tiles into slices has at most one slice per SM
// (see launch_router), any other one per tile.
static size_t max_slices(const fb_ctx* ctx) {
  const size_t tiles = static_cast<size_t>(ctx->max_tiles), sliced = static_cast<size_t>(ctx->n_sm) + 8;
  return tiles > sliced ? tiles : sliced;
}

extern "C" {

const char* fb_status_string(fb_status s) {
  switch (s) {
    case FB_OK: return "ok";
    case FB_ERR_INVALID_ARG: return "invalid argument";
    case FB_ERR_UNSUPPORTED_SHAPE: return "unsupported shape";
    case FB_ERR_CUDA: return "CUDA call failed";
    case FB_ERR_BAD_PLACEMENT: return "expert_to_slot is not a bijection";
    case FB_ERR_TIMEOUT: return "a bounded device-side wait expired";
    case FB_ERR_RANGE: return "sum of counts beyond the planner's range";
    case FB_ERR_INTERNAL: return "debug build: an output index was out of range";
  }
  return "unknown status";
}

uint64_t fb_budget_ns(uint64_t t_attn_ns, uint64_t delta_ns) {
  return t_attn_ns > delta_ns ? t_attn_ns - delta_ns : 0;
}

uint64_t fb_swap_cost_ns(const fb_budget* b, int32_t rank_a, int32_t rank_b) {
  if (!b) return 0;
  const int rpn = b->ranks_per_node;
  const int cls = (rpn <= 0 || rank_a / rpn == rank_b / rpn) ? 0 : 1;
  return uniform_cost(*b, cls);
}

fb_status fb_create(fb_ctx** out, const fb_config* cfg, int device) {
  if (!out || !cfg) return FB_ERR_INVALID_ARG;
  *out = nullptr;
  const fb_status cs = check_config(*cfg);
  if (cs != FB_OK) return cs;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) return FB_ERR_CUDA;
  DeviceGuard guard(device);
  if (!guard.ok) return FB_ERR_CUDA;
  const DeviceLimits limits = device_limits(device);
  if (!limits.usable) return FB_ERR_CUDA;
  fb_ctx* ctx = new (std::nothrow) fb_ctx();
  if (!ctx) return FB_ERR_CUDA;
  ctx->cfg = *cfg;
  ctx->device = device;
  {
    fb_status ss = setup_router_shape(ctx, limits);
    if (ss == FB_OK) ss = set_up_device(ctx, device, limits);
    if (ss != FB_OK) { delete ctx; return ss; }
  }
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
      qres != cudaDriverEntryPointSuccess || fn == nullptr) {
    delete ctx;
    return FB_ERR_CUDA;
  }
  ctx->encode = reinterpret_cast<EncodeTiledFn>(fn);
  // Everything that is zero between calls is one allocation and one memset (a context in 325 us; 337 with five of each).
  constexpr size_t kZeroWords = 3 * FB_MAX_EXPERTS + 4 * kLine;
  bool ok = dev_alloc(&ctx->counts_scratch, kZeroWords) &&
            dev_alloc(&ctx->slice_counts, max_slices(ctx) * fb::slice_row_bytes(cfg->E)) &&
            cudaMemset(ctx->counts_scratch, 0, kZeroWords * sizeof(uint32_t)) == cudaSuccess;
  if (ok) {
    ctx->totals = ctx->counts_scratch + FB_MAX_EXPERTS;
    ctx->layer_counts = ctx->totals + FB_MAX_EXPERTS;
    ctx->ticket = ctx->layer_counts + FB_MAX_EXPERTS;
    ctx->index_ticket = ctx->ticket + 2 * kLine;
    ctx->status = reinterpret_cast<int32_t*>(ctx->index_ticket + kLine);
  }
  if (!ok) { fb_destroy(ctx); return FB_ERR_CUDA; }
  *out = ctx;
  return FB_OK;
}

fb_status fb_destroy(fb_ctx* ctx) {
  if (!ctx) return FB_OK;
  DeviceGuard guard(ctx->device);
  cudaDeviceSynchronize();
  void* ptrs[] = {ctx->counts_scratch, ctx->slice_counts, ctx->st_hprev, ctx->st_H,
                  ctx->st_pi, ctx->st_pi_out, ctx->st_counts, ctx->st_swaps, ctx->st_nswaps, ctx->st_load_before,
                  ctx->st_load_after, ctx->st_ids, ctx->st_w, ctx->st_slot_offsets, ctx->st_rank_offsets,
                  ctx->st_perm, ctx->st_inv_perm, ctx->st_rank_load};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (ctx->mig_stage) cudaFree(ctx->mig_stage);
  if (ctx->mig_host) cudaFreeHost(ctx->mig_host);
  for (auto& a : ctx->attn) {
    if (a.e0) cudaEventDestroy(a.e0);
    if (a.e1) cudaEventDestroy(a.e1);
  }
  delete ctx;
  return FB_OK;
}

fb_status fb_predict_load(fb_ctx* ctx, const fb_router* router, const void* x, int32_t T, uint32_t* counts,
                          int32_t* topk_ids, float* logits, fb_stream stream_) {
  if (!ctx || !router || !router->W || !counts || T < 0) return FB_ERR_INVALID_ARG;
  if (T > ctx->cfg.T_max) return FB_ERR_UNSUPPORTED_SHAPE;
  if (T > 0 && !x) return FB_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  if (T == 0)
    return cudaMemsetAsync(counts, 0, ctx->cfg.E * sizeof(uint32_t), stream) == cudaSuccess ? FB_OK : FB_ERR_CUDA;
  return launch_router(ctx, router, x, T, fb::kModePredict, counts, topk_ids, nullptr, logits, nullptr, stream);
}

fb_status fb_plan_swaps(fb_ctx* ctx, const uint32_t* counts, const int32_t* expert_to_slot, const fb_budget* budget,
                        int32_t layer_id, int32_t* expert_to_slot_out, fb_swap* swaps, int32_t* n_swaps,
                        uint32_t* load_before, uint32_t* load_after, fb_stream stream_) {
  (void)layer_id;   // constant within a call: it leads the tie-break tuple but cannot change the order
  if (!ctx || !counts) return FB_ERR_INVALID_ARG;
  fb::PlanParams pp;
  memset(&pp, 0, sizeof(pp));
  const fb_status st = fill_plan(ctx, budget, expert_to_slot, expert_to_slot_out, swaps, n_swaps, load_before,
                                 load_after, &pp);
  if (st != FB_OK) return st;
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  return launch_plan(ctx, pp, const_cast<uint32_t*>(counts), nullptr, kAnyShare, static_cast<cudaStream_t>(stream_));   // (read only)
}

fb_status fb_predict_and_plan(fb_ctx* ctx, const fb_router* router, const void* x, int32_t T,
                              const int32_t* expert_to_slot, const fb_budget* budget, int32_t layer_id,
                              uint32_t* counts, int32_t* expert_to_slot_out, fb_swap* swaps, int32_t* n_swaps,
                              uint32_t* load_before, uint32_t* load_after, fb_stream stream_) {
  (void)layer_id;
  if (!ctx || !router || !router->W || !counts || T < 0) return FB_ERR_INVALID_ARG;
  if (T > ctx->cfg.T_max) return FB_ERR_UNSUPPORTED_SHAPE;
  if (T > 0 && !x) return FB_ERR_INVALID_ARG;
  fb::PlanParams pp;
  memset(&pp, 0, sizeof(pp));
  const fb_status st = fill_plan(ctx, budget, expert_to_slot, expert_to_slot_out, swaps, n_swaps, load_before,
                                 load_after, &pp);
  if (st != FB_OK) return st;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  if (T == 0) {
    if (cudaMemsetAsync(counts, 0, ctx->cfg.E * sizeof(uint32_t), stream) != cudaSuccess) return FB_ERR_CUDA;
    return launch_plan(ctx, pp, counts, nullptr, kAnyShare, stream);
  }
  return launch_router(ctx, router, x, T, fb::kModePredictPlan, counts, nullptr, nullptr, nullptr, &pp, stream);
}

fb_status fb_route_dispatch(fb_ctx* ctx, const fb_router* router, const void* x, int32_t T,
                            const int32_t* expert_to_slot, int32_t* topk_ids, float* topk_w, uint32_t* slot_offsets,
                            uint32_t* rank_offsets, int32_t* perm, int32_t* inv_perm, uint32_t* rank_load,
                            float* logits, fb_stream stream_) {
  if (!ctx || !router || !router->W || !expert_to_slot || !slot_offsets || !rank_offsets || !rank_load || T < 0)
    return FB_ERR_INVALID_ARG;
  if (T > ctx->cfg.T_max) return FB_ERR_UNSUPPORTED_SHAPE;
  if (T > 0 && (!x || !topk_ids || !topk_w || !perm || !inv_perm)) return FB_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  const fb_config& c = ctx->cfg;
  if (T == 0) {
    if (cudaMemsetAsync(slot_offsets, 0, (c.E + 1) * sizeof(uint32_t), stream) != cudaSuccess ||
        cudaMemsetAsync(rank_offsets, 0, (c.R + 1) * sizeof(uint32_t), stream) != cudaSuccess ||
        cudaMemsetAsync(rank_load, 0, c.R * sizeof(uint32_t), stream) != cudaSuccess)
      return FB_ERR_CUDA;
    return FB_OK;
  }
  int pieces = 1;
  const fb_status st = launch_router(ctx, router, x, T, fb::kModeDispatch, nullptr, topk_ids, topk_w, logits,
                                     nullptr, stream, nullptr, 0, &pieces);
  if (st != FB_OK) return st;
  return launch_dispatch_index(ctx, T, pieces, nullptr, nullptr, expert_to_slot, topk_ids, slot_offsets, rank_offsets,
                               perm, inv_perm, rank_load, stream);
}

fb_status fb_layer_step_observed(fb_ctx* ctx, const fb_router* router, const void* h_prev, const void* H, int32_t T,
                        const int32_t* expert_to_slot, const fb_budget* budget, int32_t layer_id,
                        uint32_t* counts, int32_t* expert_to_slot_out, fb_swap* swaps, int32_t* n_swaps,
                        uint32_t* load_before, uint32_t* load_after, int32_t* topk_ids, float* topk_w,
                        uint32_t* slot_offsets, uint32_t* rank_offsets, int32_t* perm, int32_t* inv_perm,
                        uint32_t* rank_load, int32_t* ids_early, float* logits_early, float* logits,
                                 fb_stream stream_) {
  (void)layer_id;
  if (!ctx || !router || !router->W || !counts || !slot_offsets || !rank_offsets || !rank_load || T < 0)
    return FB_ERR_INVALID_ARG;
  if (T > ctx->cfg.T_max) return FB_ERR_UNSUPPORTED_SHAPE;
  if (T > 0 && (!h_prev || !H || !topk_ids || !topk_w || !perm || !inv_perm)) return FB_ERR_INVALID_ARG;
  if (T == 0) {
    const fb_status st0 = fb_predict_and_plan(ctx, router, h_prev, 0, expert_to_slot, budget, layer_id, counts,
                                              expert_to_slot_out, swaps, n_swaps, load_before, load_after, stream_);
    if (st0 != FB_OK) return st0;
    return fb_route_dispatch(ctx, router, H, 0, expert_to_slot_out, topk_ids, topk_w, slot_offsets, rank_offsets,
                             perm, inv_perm, rank_load, nullptr, stream_);
  }
  fb::PlanParams pp;
  memset(&pp, 0, sizeof(pp));
  fb_status st = fill_plan(ctx, budget, expert_to_slot, expert_to_slot_out, swaps, n_swaps, load_before, load_after,
                           &pp);
  if (st != FB_OK) return st;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  // one launch for both router passes; the dispatch index needs the new placement and follows
  int pieces = 1;
  bool deferred = false;
  st = launch_router(ctx, router, h_prev, T, fb::kModeLayer, counts, topk_ids, topk_w, logits, &pp, stream, H, 0, &pieces,
                     &deferred, ids_early, logits_early);
  if (st != FB_OK) return st;
  return launch_dispatch_index(ctx, T, pieces, deferred ? &pp : nullptr, counts,
                               deferred ? expert_to_slot : expert_to_slot_out, topk_ids, slot_offsets, rank_offsets, perm,
                               inv_perm, rank_load, stream);
}

fb_status fb_layer_step(fb_ctx* ctx, const fb_router* router, const void* h_prev, const void* H, int32_t T,
                        const int32_t* expert_to_slot, const fb_budget* budget, int32_t layer_id,
                        uint32_t* counts, int32_t* expert_to_slot_out, fb_swap* swaps, int32_t* n_swaps,
                        uint32_t* load_before, uint32_t* load_after, int32_t* topk_ids, float* topk_w,
                        uint32_t* slot_offsets, uint32_t* rank_offsets, int32_t* perm, int32_t* inv_perm,
                        uint32_t* rank_load, fb_stream stream) {
  return fb_layer_step_observed(ctx, router, h_prev, H, T, expert_to_slot, budget, layer_id, counts, expert_to_slot_out,
                                swaps, n_swaps, load_before, load_after, topk_ids, topk_w, slot_offsets, rank_offsets,
                                perm, inv_perm, rank_load, nullptr, nullptr, nullptr, stream);
}

fb_status fb_layer_step_host(fb_ctx* ctx, const fb_router* router, const void* h_prev_host, const void* H_host,
                             int32_t T, const int32_t* expert_to_slot_host, const fb_budget* budget,
                             int32_t layer_id, uint32_t* counts, int32_t* expert_to_slot_out, fb_swap* swaps,
                             int32_t* n_swaps, uint32_t* load_before, uint32_t* load_after, int32_t* topk_ids,
                             float* topk_w, uint32_t* slot_offsets, uint32_t* rank_offsets, int32_t* perm,
                             int32_t* inv_perm, uint32_t* rank_load, fb_stream stream_) {
  if (!ctx || !router || !expert_to_slot_host || !budget || T < 0) return FB_ERR_INVALID_ARG;
  if (T > ctx->cfg.T_max) return FB_ERR_UNSUPPORTED_SHAPE;
  if (T > 0 && (!h_prev_host || !H_host)) return FB_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  const fb_config& c = ctx->cfg;
  const size_t Tm = static_cast<size_t>(c.T_max), E = c.E, R = c.R, k = c.k;
  if (!ctx->staged) {
    const size_t act = Tm * c.d * 2;
    bool ok = cudaMalloc(&ctx->st_hprev, act ? act : 16) == cudaSuccess &&
              cudaMalloc(&ctx->st_H, act ? act : 16) == cudaSuccess;
    ok = ok && dev_alloc(&ctx->st_pi, E) && dev_alloc(&ctx->st_pi_out, E) && dev_alloc(&ctx->st_counts, E) &&
         dev_alloc(&ctx->st_swaps, E / 2 + 1) && dev_alloc(&ctx->st_nswaps, 1) &&
         dev_alloc(&ctx->st_load_before, R) && dev_alloc(&ctx->st_load_after, R) &&
         dev_alloc(&ctx->st_ids, Tm * k) && dev_alloc(&ctx->st_w, Tm * k) &&
         dev_alloc(&ctx->st_slot_offsets, E + 1) && dev_alloc(&ctx->st_rank_offsets, R + 1) &&
         dev_alloc(&ctx->st_perm, Tm * k) && dev_alloc(&ctx->st_inv_perm, Tm * k) &&
         dev_alloc(&ctx->st_rank_load, R);
    if (!ok) return FB_ERR_CUDA;
    ctx->staged = true;
  }
  const size_t act_bytes = static_cast<size_t>(T) * c.d * 2;
  const size_t n_assign = static_cast<size_t>(T) * k;
  bool ok = true;
  if (T > 0) {
    ok = ok && cudaMemcpyAsync(ctx->st_hprev, h_prev_host, act_bytes, cudaMemcpyHostToDevice, stream) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(ctx->st_H, H_host, act_bytes, cudaMemcpyHostToDevice, stream) == cudaSuccess;
  }
  ok = ok && cudaMemcpyAsync(ctx->st_pi, expert_to_slot_host, E * sizeof(int32_t), cudaMemcpyHostToDevice, stream) ==
                 cudaSuccess;
  if (!ok) return FB_ERR_CUDA;
  const fb_status st = fb_layer_step(ctx, router, ctx->st_hprev, ctx->st_H, T, ctx->st_pi, budget, layer_id,
                                     ctx->st_counts, ctx->st_pi_out, ctx->st_swaps, ctx->st_nswaps,
                                     ctx->st_load_before, ctx->st_load_after, ctx->st_ids, ctx->st_w,
                                     ctx->st_slot_offsets, ctx->st_rank_offsets, ctx->st_perm, ctx->st_inv_perm,
                                     ctx->st_rank_load, stream);
  if (st != FB_OK) return st;
  auto back = [&](void* dst, const void* src, size_t bytes) {
    if (dst && bytes) ok = ok && cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, stream) == cudaSuccess;
  };
  back(counts, ctx->st_counts, E * sizeof(uint32_t));
  back(expert_to_slot_out, ctx->st_pi_out, E * sizeof(int32_t));
  back(swaps, ctx->st_swaps, budget->max_swaps * sizeof(fb_swap));
  back(n_swaps, ctx->st_nswaps, sizeof(int32_t));
  back(load_before, ctx->st_load_before, R * sizeof(uint32_t));
  back(load_after, ctx->st_load_after, R * sizeof(uint32_t));
  back(topk_ids, ctx->st_ids, n_assign * sizeof(int32_t));
  back(topk_w, ctx->st_w, n_assign * sizeof(float));
  back(slot_offsets, ctx->st_slot_offsets, (E + 1) * sizeof(uint32_t));
  back(rank_offsets, ctx->st_rank_offsets, (R + 1) * sizeof(uint32_t));
  back(perm, ctx->st_perm, n_assign * sizeof(int32_t));
  back(inv_perm, ctx->st_inv_perm, n_assign * sizeof(int32_t));
  back(rank_load, ctx->st_rank_load, R * sizeof(uint32_t));
  if (!ok) return FB_ERR_CUDA;
  return cudaStreamSynchronize(stream) == cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_device_status(fb_ctx* ctx, int32_t* word, fb_stream stream_) {
  if (!ctx || !word) return FB_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  if (cudaStreamSynchronize(stream) != cudaSuccess) return FB_ERR_CUDA;
  if (cudaMemcpy(word, ctx->status, sizeof(int32_t), cudaMemcpyDeviceToHost) != cudaSuccess) return FB_ERR_CUDA;
  if (*word != 0) {
    if (cudaMemset(ctx->status, 0, sizeof(int32_t)) != cudaSuccess) return FB_ERR_CUDA;
  }
  return FB_OK;
}

uint64_t fb_launch_count(const fb_ctx* ctx) { return ctx ? ctx->launches : 0; }

fb_status fb_apply_swaps(void* slot_weights, uint64_t expert_bytes, int32_t E, const int32_t* expert_to_slot,
                         const fb_swap* swaps, const int32_t* n_swaps, int32_t max_swaps, int32_t* status_word,
                         fb_stream stream_) {
  if (E < 1 || E > FB_MAX_EXPERTS || max_swaps < 0 || expert_bytes % 16 != 0) return FB_ERR_INVALID_ARG;
  if (max_swaps == 0 || expert_bytes == 0) return FB_OK;
  if (!slot_weights || !expert_to_slot || !swaps || !n_swaps) return FB_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(slot_weights) % 16 != 0) return FB_ERR_INVALID_ARG;
  // the launch goes to the device that holds the weights, whichever device is current
  const int device = device_of(slot_weights);
  if (device < 0) return FB_ERR_INVALID_ARG;
  DeviceGuard guard(device);
  if (!guard.ok) return FB_ERR_CUDA;
  fb::MigrateParams mp;
  mp.slot_weights = static_cast<uint8_t*>(slot_weights);
  mp.expert_bytes = expert_bytes;
  mp.E = E;
  mp.expert_to_slot = expert_to_slot;
  mp.swaps = swaps;
  mp.n_swaps = n_swaps;
  mp.status = status_word;
  mp.max_swaps = max_swaps;
  mp.copy_bytes = expert_bytes;
  const uint64_t per_piece = static_cast<uint64_t>(fb::kMigrateThreads) * fb::kMigrateUnroll * 16;
  uint64_t units = (expert_bytes + per_piece - 1) / per_piece * static_cast<uint64_t>(max_swaps);
  if (units > fb::kMigrateBlocks) units = fb::kMigrateBlocks;
  const dim3 grid(static_cast<unsigned>(units), 1, 1);
  fb::fb_swap_weights_kernel<<<grid, fb::kMigrateThreads, 0, static_cast<cudaStream_t>(stream_)>>>(mp);
  return cudaGetLastError() == cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_fit_cost_model(uint64_t t_small_ns, uint64_t t_large_ns, uint64_t bytes_small, uint64_t bytes_large,
                            uint64_t* alpha_ns, uint64_t* fs_per_byte) {
  if (!alpha_ns || !fs_per_byte || bytes_large <= bytes_small || t_large_ns <= t_small_ns) return FB_ERR_INVALID_ARG;
  const unsigned __int128 d_bytes = static_cast<unsigned __int128>(2) * (bytes_large - bytes_small);
  const unsigned __int128 d_t = t_large_ns - t_small_ns;
  const unsigned __int128 fs = (d_t * 1000000u + d_bytes - 1) / d_bytes;             // 1 / beta, rounded up
  if (fs > ~static_cast<uint64_t>(0)) return FB_ERR_RANGE;
  // alpha = t_small - 2 S_small * d_t / d_bytes, rounded down, not below zero
  const unsigned __int128 lhs = static_cast<unsigned __int128>(t_small_ns) * d_bytes;
  const unsigned __int128 rhs = static_cast<unsigned __int128>(2) * bytes_small * d_t;
  *alpha_ns = lhs > rhs ? static_cast<uint64_t>((lhs - rhs) / d_bytes) : 0;
  *fs_per_byte = static_cast<uint64_t>(fs);
  return FB_OK;
}

fb_status fb_calibrate_exchange(void* slot_weights, uint64_t bytes_small, uint64_t bytes_large, int32_t reps,
                                uint64_t* alpha_ns, uint64_t* fs_per_byte, uint64_t* t_small_ns_out,
                                uint64_t* t_large_ns_out, fb_stream stream_) {
  if (!slot_weights || !alpha_ns || !fs_per_byte || reps < 1 || reps > 1000 || bytes_small == 0 ||
      bytes_small % 16 != 0 || bytes_large % 16 != 0 || bytes_large <= bytes_small)
    return FB_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  const int device = device_of(slot_weights);
  if (device < 0) return FB_ERR_INVALID_ARG;
  DeviceGuard guard(device);
  if (!guard.ok) return FB_ERR_CUDA;
  // a one-swap plan over two slots: constant data of the library image on this device
  const int32_t* plan = nullptr;                 // [pi: 2][swap: 4][n: 1]
  if (cudaGetSymbolAddress(reinterpret_cast<void**>(const_cast<int32_t**>(&plan)), g_calibration_plan) !=
          cudaSuccess || plan == nullptr)
    return FB_ERR_CUDA;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  bool ok = cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess;
  uint64_t t_ns[2] = {0, 0};
  const uint64_t sizes[2] = {bytes_small, bytes_large};
  for (int which = 0; which < 2 && ok; ++which) {
    // the two images lie bytes_large apart for both sizes: the same addresses are warm in both runs
    float best = 0.0f;
    for (int r = 0; r < reps + 2 && ok; ++r) {
      ok = cudaEventRecord(e0, stream) == cudaSuccess;
      fb::MigrateParams mp;
      mp.slot_weights = static_cast<uint8_t*>(slot_weights);
      mp.expert_bytes = bytes_large;             // slot stride
      mp.E = 2;
      mp.expert_to_slot = plan;
      mp.swaps = reinterpret_cast<const fb_swap*>(plan + 2);
      mp.n_swaps = plan + 6;
      mp.max_swaps = 1;
      mp.status = nullptr;
      mp.copy_bytes = sizes[which];
      const uint64_t per_piece = static_cast<uint64_t>(fb::kMigrateThreads) * fb::kMigrateUnroll * 16;
      uint64_t units = (sizes[which] + per_piece - 1) / per_piece;
      if (units > fb::kMigrateBlocks) units = fb::kMigrateBlocks;
      fb::fb_swap_weights_kernel<<<static_cast<unsigned>(units), fb::kMigrateThreads, 0, stream>>>(mp);
      ok = ok && cudaEventRecord(e1, stream) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess;
      float ms = 0.0f;
      ok = ok && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
      if (r >= 2 && (best == 0.0f || ms < best)) best = ms;          // first two runs warm up; keep the fastest
    }
    t_ns[which] = static_cast<uint64_t>(best * 1e6f);
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (!ok) return FB_ERR_CUDA;
  if (t_small_ns_out) *t_small_ns_out = t_ns[0];
  if (t_large_ns_out) *t_large_ns_out = t_ns[1];
  return fb_fit_cost_model(t_ns[0], t_ns[1], bytes_small, bytes_large, alpha_ns, fs_per_byte);
}

fb_status fb_apply_swaps_staged(fb_ctx* ctx, void* slot_weights, uint64_t expert_bytes, const int32_t* expert_to_slot,
                                const fb_swap* swaps, const int32_t* n_swaps, int32_t max_swaps,
                                uint64_t staging_bytes, fb_stream plan_stream_, fb_stream copy_stream_) {
  if (!ctx || max_swaps < 0 || max_swaps > FB_MAX_EXPERTS / 2) return FB_ERR_INVALID_ARG;
  if (max_swaps == 0 || expert_bytes == 0) return FB_OK;
  if (!slot_weights || !expert_to_slot || !swaps || !n_swaps) return FB_ERR_INVALID_ARG;
  cudaStream_t plan_stream = static_cast<cudaStream_t>(plan_stream_);
  cudaStream_t copy_stream = static_cast<cudaStream_t>(copy_stream_);
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  const int E = ctx->cfg.E;
  if (staging_bytes == 0 || staging_bytes > expert_bytes) staging_bytes = expert_bytes;
  // host copy of the plan: [n_swaps][swaps: max_swaps][placement: E]
  const size_t host_bytes = sizeof(int32_t) * (1 + 4 * static_cast<size_t>(FB_MAX_EXPERTS / 2) + FB_MAX_EXPERTS);
  if (!ctx->mig_host && cudaMallocHost(&ctx->mig_host, host_bytes) != cudaSuccess) return FB_ERR_CUDA;
  if (ctx->mig_stage_bytes < staging_bytes) {
    if (ctx->mig_stage) { cudaStreamSynchronize(copy_stream); cudaFree(ctx->mig_stage); ctx->mig_stage = nullptr; }
    if (cudaMalloc(&ctx->mig_stage, staging_bytes) != cudaSuccess) { ctx->mig_stage_bytes = 0; return FB_ERR_CUDA; }
    ctx->mig_stage_bytes = staging_bytes;
  }
  int32_t* h_n = static_cast<int32_t*>(ctx->mig_host);
  fb_swap* h_swaps = reinterpret_cast<fb_swap*>(h_n + 1);
  int32_t* h_pi = h_n + 1 + 4 * (FB_MAX_EXPERTS / 2);
  bool ok = cudaMemcpyAsync(h_n, n_swaps, sizeof(int32_t), cudaMemcpyDeviceToHost, plan_stream) == cudaSuccess &&
            cudaMemcpyAsync(h_swaps, swaps, sizeof(fb_swap) * max_swaps, cudaMemcpyDeviceToHost, plan_stream) ==
                cudaSuccess &&
            cudaMemcpyAsync(h_pi, expert_to_slot, sizeof(int32_t) * E, cudaMemcpyDeviceToHost, plan_stream) ==
                cudaSuccess &&
            cudaStreamSynchronize(plan_stream) == cudaSuccess;       // the host needs the plan to issue the copies
  if (!ok) return FB_ERR_CUDA;
  const int n = *h_n;
  if (n < 0 || n > max_swaps) return FB_ERR_RANGE;
  uint8_t* base = static_cast<uint8_t*>(slot_weights);
  for (int i = 0; i < n; ++i) {
    const int ea = h_swaps[i].expert_src, eb = h_swaps[i].expert_dst;
    if (ea < 0 || ea >= E || eb < 0 || eb >= E || ea == eb) return FB_ERR_RANGE;
    const int pa = h_pi[ea], pb = h_pi[eb];
    if (pa < 0 || pa >= E || pb < 0 || pb >= E || pa == pb) return FB_ERR_BAD_PLACEMENT;
    uint8_t* A = base + static_cast<uint64_t>(pa) * expert_bytes;
    uint8_t* Bp = base + static_cast<uint64_t>(pb) * expert_bytes;
    // pairwise exchange through the bounded staging buffer, one piece at a time
    for (uint64_t off = 0; off < expert_bytes; off += staging_bytes) {
      const uint64_t len = expert_bytes - off < staging_bytes ? expert_bytes - off : staging_bytes;
      ok = ok && cudaMemcpyAsync(ctx->mig_stage, A + off, len, cudaMemcpyDeviceToDevice, copy_stream) == cudaSuccess &&
           cudaMemcpyAsync(A + off, Bp + off, len, cudaMemcpyDeviceToDevice, copy_stream) == cudaSuccess &&
           cudaMemcpyAsync(Bp + off, ctx->mig_stage, len, cudaMemcpyDeviceToDevice, copy_stream) == cudaSuccess;
    }
  }
  return ok ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_row_cosine_mean(const void* a, const void* b, int64_t rows, int32_t n, int32_t dtype,
                             double* row_scratch, double* mean_out, fb_stream stream_) {
  if (rows < 0 || n <= 0 || (dtype != FB_DTYPE_BF16 && dtype != FB_DTYPE_F32) || !mean_out) return FB_ERR_INVALID_ARG;
  if (rows > 0 && (!a || !b || !row_scratch)) return FB_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  cudaError_t err = cudaSuccess;
  // One launch in all practice: a grid holds 2^31 - 1 blocks, more rows than a part's go in several.
  constexpr int64_t kPart = int64_t{1} << 31;
  for (int64_t r0 = 0; r0 < rows && err == cudaSuccess; r0 += kPart) {
    const int64_t part = rows - r0 < kPart ? rows - r0 : kPart;
    const int blocks = static_cast<int>((part + fb::kCosineWarpsPerBlock - 1) / fb::kCosineWarpsPerBlock);
    if (dtype == FB_DTYPE_BF16)
      err = launch_dependent(fb::fb_row_cosine_kernel<__nv_bfloat16>, blocks, 32 * fb::kCosineWarpsPerBlock, kAnyShare, stream,
                             static_cast<const __nv_bfloat16*>(a) + r0 * n, static_cast<const __nv_bfloat16*>(b) + r0 * n,
                             static_cast<long long>(part), n, row_scratch + r0);
    else
      err = launch_dependent(fb::fb_row_cosine_kernel<float>, blocks, 32 * fb::kCosineWarpsPerBlock, kAnyShare, stream,
                             static_cast<const float*>(a) + r0 * n, static_cast<const float*>(b) + r0 * n,
                             static_cast<long long>(part), n, row_scratch + r0);
  }
  if (err == cudaSuccess)
    err = launch_dependent(fb::fb_mean_kernel, 1, fb::kMeanThreads, kAnyShare, stream, row_scratch, static_cast<long long>(rows), mean_out);
  return err == cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_topk_hits(const int32_t* ids_a, const int32_t* ids_b, int32_t T, int32_t k, uint32_t* hits_out,
                       fb_stream stream_) {
  if (T < 0 || k < 1 || k > FB_MAX_TOPK || !hits_out || (T > 0 && (!ids_a || !ids_b))) return FB_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  return launch_dependent(fb::fb_topk_hits_kernel, fb::kHitsBlocks, fb::kHitsThreads, kAnyShare, stream, ids_a, ids_b, T, k, hits_out) ==
                 cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_prediction_quality(const void* h_prev, const void* H, const float* z_early, const float* z,
                                const int32_t* ids_early, const int32_t* ids, int32_t T, int32_t d, int32_t E, int32_t k,
                                double* row_scratch, double* metrics_out, fb_stream stream_) {
  if (T < 0 || d <= 0 || E <= 0 || k < 1 || k > FB_MAX_TOPK || !metrics_out) return FB_ERR_INVALID_ARG;
  if (T > 0 && (!h_prev || !H || !z_early || !z || !ids_early || !ids || !row_scratch)) return FB_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  fb::QualityParams qp;
  qp.h_prev = static_cast<const __nv_bfloat16*>(h_prev);
  qp.h = static_cast<const __nv_bfloat16*>(H);
  qp.z_early = z_early;
  qp.z = z;
  qp.ids_early = ids_early;
  qp.ids = ids;
  qp.T = T; qp.d = d; qp.E = E; qp.k = k;
  qp.rows = row_scratch;
  qp.out = metrics_out;
  cudaError_t err = cudaSuccess;
  if (T > 0)
    err = launch_dependent(fb::fb_quality_rows_kernel, (T - 1) / fb::kCosineWarpsPerBlock + 1,
                           32 * fb::kCosineWarpsPerBlock, kAnyShare, stream, qp);
  if (err == cudaSuccess) err = launch_dependent(fb::fb_quality_sums_kernel, fb::kQualityBlocks, fb::kMeanThreads, kAnyShare, stream, qp);
  return err == cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_set_split(fb_ctx* ctx, int32_t mode, int32_t owner_bias_kblocks) {
  if (!ctx || (mode != 0 && mode != 1) || owner_bias_kblocks < -1 || owner_bias_kblocks > 1024) return FB_ERR_INVALID_ARG;
  ctx->split_mode = mode;      // (the pieces of a tile's k-range are equal: there is no owner to favour)
  return FB_OK;
}

fb_status fb_staged_row_layout(const fb_config* cfg, int32_t* row_words, int32_t* stored_at, int32_t* read_at) {
  if (!cfg || !row_words || !stored_at || !read_at) return FB_ERR_INVALID_ARG;
  const fb_status cs = check_config(*cfg);
  if (cs != FB_OK) return cs;
  fb::RouterParams g;
  memset(&g, 0, sizeof(g));
  g.E = cfg->E;
  g.N = (cfg->E + 15) / 16 * 16;
  fb::gate_layout(cfg->E, cfg->gate, cfg->n_group, cfg->topk_group, &g);
  *row_words = fb::staging_stride(g.N);
  for (int c = 0; c < FB_MAX_EXPERTS; ++c) {
    stored_at[c] = c < g.N ? fb::quad_word(g, c / 4) + c % 4 : -1;
    read_at[c] = -1;
  }
  for (int lane = 0; lane < 32; ++lane) {
    const fb::LaneColumns lc = fb::lane_columns(g, lane);
    for (int j = 0; j < lc.n; ++j) read_at[lc.c0 + j] = lc.word + (g.two_vectors ? j / 4 * 128 + j % 4 : j);
  }
  return FB_OK;
}

fb_status fb_fail_launch(fb_ctx* ctx, int32_t nth) {
  if (!ctx || nth < 0) return FB_ERR_INVALID_ARG;
  ctx->fail_launch = nth;
  return FB_OK;
}

fb_status fb_set_stage_limit(fb_ctx* ctx, int32_t stages) {
  if (!ctx || stages < 0 || stages == 1) return FB_ERR_INVALID_ARG;
  ctx->stage_limit = stages;
  return FB_OK;
}

fb_status fb_set_pair_limit(fb_ctx* ctx, int32_t pairs) {
  if (!ctx || pairs < 0) return FB_ERR_INVALID_ARG;
  ctx->pair_limit = pairs;
  return FB_OK;
}

fb_status fb_time_next_router_launch(fb_ctx* ctx, void* event_before, void* event_after) {
  if (!ctx) return FB_ERR_INVALID_ARG;
  ctx->ev_before = static_cast<cudaEvent_t>(event_before);
  ctx->ev_after = static_cast<cudaEvent_t>(event_after);
  return FB_OK;
}

fb_status fb_router_floor(fb_ctx* ctx, const fb_router* router, const void* x, int32_t T, int32_t what,
                          fb_stream stream_) {
  if (!ctx || !router || !router->W || !x || T <= 0 || (what != 1 && what != 2)) return FB_ERR_INVALID_ARG;
  if (T > ctx->cfg.T_max) return FB_ERR_UNSUPPORTED_SHAPE;
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  return launch_router(ctx, router, x, T, fb::kModePredict, nullptr, nullptr, nullptr, nullptr, nullptr,
                       static_cast<cudaStream_t>(stream_), nullptr, what);
}

int32_t fb_max_pairs(const fb_ctx* ctx) { return ctx && ctx->ranking[0] ? ctx->max_clusters[1] : 0; }

fb_status fb_dispatch_slot_counts(fb_ctx* ctx, const uint32_t* slot_offsets, uint32_t* slot_counts, fb_stream stream_) {
  if (!ctx || !slot_offsets || !slot_counts) return FB_ERR_INVALID_ARG;
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  const cudaError_t err = launch_counted(ctx, fb::fb_slot_counts_kernel, 1, FB_MAX_EXPERTS, kAnyShare, static_cast<cudaStream_t>(stream_),
                                         slot_offsets, ctx->cfg.E, slot_counts);
  return err == cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_dispatch_globalize(fb_ctx* ctx, int32_t T_local, int32_t world, int32_t rank,
                                const uint32_t* slot_counts_all, const uint32_t* slot_offsets_local,
                                const int32_t* topk_ids, const int32_t* expert_to_slot, int32_t* inv_perm,
                                uint32_t* slot_offsets, uint32_t* rank_offsets, uint32_t* rank_load,
                                fb_stream stream_) {
  if (!ctx || T_local < 0 || world < 1 || world > 4096 || rank < 0 || rank >= world || !slot_counts_all ||
      !slot_offsets_local || !expert_to_slot || !slot_offsets || !rank_offsets || !rank_load)
    return FB_ERR_INVALID_ARG;
  if (T_local > ctx->cfg.T_max) return FB_ERR_UNSUPPORTED_SHAPE;
  if (T_local > 0 && (!topk_ids || !inv_perm)) return FB_ERR_INVALID_ARG;
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  fb::GlobalizeParams gp;
  gp.T = T_local; gp.k = ctx->cfg.k; gp.E = ctx->cfg.E; gp.R = ctx->cfg.R; gp.world = world; gp.rank = rank;
  gp.per_rank = ctx->cfg.E / ctx->cfg.R;
  gp.counts_all = slot_counts_all; gp.local_offsets = slot_offsets_local; gp.topk_ids = topk_ids;
  gp.expert_to_slot = expert_to_slot; gp.inv_perm = inv_perm;
  gp.slot_offsets = slot_offsets; gp.rank_offsets = rank_offsets; gp.rank_load = rank_load;
  const long long n = static_cast<long long>(T_local) * ctx->cfg.k;
  long long blocks = (n + fb::kGlobalizeThreads - 1) / fb::kGlobalizeThreads;
  if (blocks < 1) blocks = 1;
  if (blocks > 4 * ctx->n_sm) blocks = 4 * ctx->n_sm;
  const cudaError_t err = launch_counted(ctx, fb::fb_dispatch_globalize_kernel, static_cast<int>(blocks), fb::kGlobalizeThreads, kAnyShare,
                                         static_cast<cudaStream_t>(stream_), gp);
  return err == cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_attention_begin(fb_ctx* ctx, int32_t layer_id, int32_t attn_type, fb_stream stream_) {
  if (!ctx || attn_type < 0 || attn_type >= FB_MAX_ATTENTION_TYPES || layer_id < 0) return FB_ERR_INVALID_ARG;
  fb_ctx::AttnSlot& a = ctx->attn[attn_type];
  if (a.layer >= 0) return FB_OK;                      // this type already has its r(l)
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  if (!a.e0 && cudaEventCreate(&a.e0) != cudaSuccess) return FB_ERR_CUDA;
  if (!a.e1 && cudaEventCreate(&a.e1) != cudaSuccess) return FB_ERR_CUDA;
  if (cudaEventRecord(a.e0, static_cast<cudaStream_t>(stream_)) != cudaSuccess) return FB_ERR_CUDA;
  a.layer = layer_id;
  a.open = true;
  return FB_OK;
}

fb_status fb_attention_end(fb_ctx* ctx, int32_t layer_id, int32_t attn_type, fb_stream stream_) {
  if (!ctx || attn_type < 0 || attn_type >= FB_MAX_ATTENTION_TYPES || layer_id < 0) return FB_ERR_INVALID_ARG;
  fb_ctx::AttnSlot& a = ctx->attn[attn_type];
  if (!a.open || a.layer != layer_id) return FB_OK;    // not the layer being measured
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  if (cudaEventRecord(a.e1, static_cast<cudaStream_t>(stream_)) != cudaSuccess) return FB_ERR_CUDA;
  a.open = false;
  a.pending = true;
  return FB_OK;
}

fb_status fb_layer_budget_ns(fb_ctx* ctx, int32_t attn_type, uint64_t delta_ns, uint64_t* budget_ns,
                             int32_t* profiled_layer) {
  if (!ctx || !budget_ns || attn_type < 0 || attn_type >= FB_MAX_ATTENTION_TYPES) return FB_ERR_INVALID_ARG;
  fb_ctx::AttnSlot& a = ctx->attn[attn_type];
  if (a.pending) {
    DeviceGuard guard(ctx->device);
    if (!guard.ok) return FB_ERR_CUDA;
    float ms = 0.0f;
    if (cudaEventSynchronize(a.e1) != cudaSuccess || cudaEventElapsedTime(&ms, a.e0, a.e1) != cudaSuccess)
      return FB_ERR_CUDA;
    a.t_ns = static_cast<uint64_t>(static_cast<double>(ms) * 1e6 + 0.5);
    a.pending = false;
    a.has_time = true;
  }
  if (!a.has_time) return FB_ERR_INVALID_ARG;          // never profiled (or the region is still open)
  *budget_ns = fb_budget_ns(a.t_ns, delta_ns);         // Eq. 10
  if (profiled_layer) *profiled_layer = a.layer;
  return FB_OK;
}

fb_status fb_attention_set_time_ns(fb_ctx* ctx, int32_t attn_type, int32_t layer_id, uint64_t t_attn_ns) {
  if (!ctx || attn_type < 0 || attn_type >= FB_MAX_ATTENTION_TYPES || layer_id < 0) return FB_ERR_INVALID_ARG;
  fb_ctx::AttnSlot& a = ctx->attn[attn_type];
  a.layer = layer_id;
  a.t_ns = t_attn_ns;
  a.open = a.pending = false;
  a.has_time = true;
  return FB_OK;
}

fb_status fb_attention_reset(fb_ctx* ctx) {
  if (!ctx) return FB_ERR_INVALID_ARG;
  for (auto& a : ctx->attn) { a.layer = -1; a.open = a.pending = a.has_time = false; a.t_ns = 0; }
  return FB_OK;
}

fb_status fb_standin_attention(float* out, int32_t blocks, int32_t iters, fb_stream stream_) {
  if (!out || blocks < 1 || blocks > 1024 || iters < 0 || iters > (1 << 24)) return FB_ERR_INVALID_ARG;
  const int device = device_of(out);
  if (device < 0) return FB_ERR_INVALID_ARG;
  DeviceGuard guard(device);
  if (!guard.ok) return FB_ERR_CUDA;
  static bool raised[64] = {};
  if (device < 64 && !raised[device]) {
    if (cudaFuncSetAttribute(reinterpret_cast<const void*>(fb::fb_standin_attention_kernel),
                             cudaFuncAttributeMaxDynamicSharedMemorySize, fb::kStandinSmemBytes) != cudaSuccess)
      return FB_ERR_CUDA;
    raised[device] = true;
  }
  fb::fb_standin_attention_kernel<<<static_cast<unsigned>(blocks), fb::kStandinThreads, fb::kStandinSmemBytes,
                                    static_cast<cudaStream_t>(stream_)>>>(out, iters);
  return cudaGetLastError() == cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_clock_probe(uint64_t* samples, int32_t n, uint32_t period_ns, fb_stream stream_) {
  // bounded by construction: at most 65536 samples, at most 100 us apart
  if (!samples || n < 1 || n > 65536 || period_ns > 100000) return FB_ERR_INVALID_ARG;
  const int device = device_of(samples);
  if (device < 0) return FB_ERR_INVALID_ARG;
  DeviceGuard guard(device);
  if (!guard.ok) return FB_ERR_CUDA;
  // The split between L1 and shared memory is a per-SM setting that only changes while the SM is
  // idle: a resident block of a kernel that prefers a small shared-memory share would keep the
  // router kernel's blocks (over 200 KB of shared memory each) off its SM for as long as it runs.
  static bool carveout_set[64] = {};
  if (device < 64 && !carveout_set[device]) {
    if (cudaFuncSetAttribute(reinterpret_cast<const void*>(fb::fb_clock_probe_kernel),
                             cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess)
      return FB_ERR_CUDA;
    carveout_set[device] = true;
  }
  fb::fb_clock_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream_)>>>(
      reinterpret_cast<unsigned long long*>(samples), n, period_ns);
  return cudaGetLastError() == cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_set_stamp_buffer(fb_ctx* ctx, uint64_t* stamps) {
  if (!ctx) return FB_ERR_INVALID_ARG;
#ifdef FB_TIMING
  ctx->stamps = reinterpret_cast<unsigned long long*>(stamps);
  return FB_OK;
#else
  (void)stamps;
  return FB_ERR_UNSUPPORTED_SHAPE;      // this build carries no stamp code
#endif
}

static fb_status wait_selftest(fb_ctx* ctx, uint64_t limit_ns, int32_t steps, uint64_t* waited_ns, fb_stream stream_) {
  DeviceGuard guard(ctx->device);
  if (!guard.ok) return FB_ERR_CUDA;
  fb::fb_wait_selftest_kernel<<<1, 64, 0, static_cast<cudaStream_t>(stream_)>>>(limit_ns, steps, ctx->status, waited_ns);
  ++ctx->launches;
  return cudaGetLastError() == cudaSuccess ? FB_OK : FB_ERR_CUDA;
}

fb_status fb_selftest_wait_timeout(fb_ctx* ctx, uint64_t limit_ns, uint64_t* waited_ns, fb_stream stream) {
  if (!ctx || limit_ns == 0 || limit_ns > 100ull * 1000 * 1000) return FB_ERR_INVALID_ARG;
  return wait_selftest(ctx, limit_ns, 0, waited_ns, stream);
}

fb_status fb_selftest_wait_progress(fb_ctx* ctx, uint64_t limit_ns, int32_t steps, uint64_t* waited_ns, fb_stream stream) {
  // half a second at most
  if (!ctx || limit_ns == 0 || limit_ns > 10ull * 1000 * 1000 || steps < 1 || steps > 100) return FB_ERR_INVALID_ARG;
  return wait_selftest(ctx, limit_ns, steps, waited_ns, stream);
}

uint64_t fb_persistent_launch_count(const fb_ctx* ctx) { return ctx ? ctx->persistent_launches : 0; }

}  // extern "C"

// ---------------------------------------------------------------------------------
// fb_predict_load_static: the prediction pass for callers that must not allocate.
// Its scratch (the cross-block histogram, the finished-block ticket and a status word)
// lives in a fixed array inside the library image instead of in an fb_ctx.
// ---------------------------------------------------------------------------------
namespace {

constexpr int kStaticScratchWords = FB_STATIC_MAX_EXPERTS + 64;
constexpr int kStaticMaxDevices = 64;

// Every GPU that loads the library holds this array until the process exits.
static __device__ __align__(256) uint32_t g_static_scratch[kStaticScratchWords];

struct StaticState {
  bool ready = false;
  uint32_t* scratch = nullptr;      // device address of g_static_scratch on this device
  fb_ctx ctx;                       // host-side launch state only; owns no device memory
};
StaticState g_static_state[kStaticMaxDevices];

}  // namespace

extern "C" fb_status fb_predict_load_static(const fb_config* cfg, int device, const fb_router* router,
                                            const void* x, int32_t T, uint32_t* counts, int32_t* topk_ids,
                                            int32_t* status_word, fb_stream stream_) {
  if (!cfg || !router || !router->W || !counts || T < 0) return FB_ERR_INVALID_ARG;
  if (cfg->E > FB_STATIC_MAX_EXPERTS) return FB_ERR_UNSUPPORTED_SHAPE;   // scratch array too small
  const fb_status cs = check_config(*cfg);
  if (cs != FB_OK) return cs;
  if (T > cfg->T_max) return FB_ERR_UNSUPPORTED_SHAPE;
  if (T > 0 && !x) return FB_ERR_INVALID_ARG;
  if (device < 0 || device >= kStaticMaxDevices) return FB_ERR_INVALID_ARG;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  DeviceGuard guard(device);
  if (!guard.ok) return FB_ERR_CUDA;
  StaticState& st = g_static_state[device];
  if (!st.ready) {
    // One-time set-up for this device, with the device current.  In host code the name
    // of a __device__ array is only a handle: the address a kernel can use has to be
    // asked for.
    if (!device_limits(device).usable) return FB_ERR_CUDA;
    void* addr = nullptr;
    if (cudaGetSymbolAddress(&addr, g_static_scratch) != cudaSuccess || addr == nullptr) return FB_ERR_CUDA;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess || fn == nullptr)
      return FB_ERR_CUDA;
    st.scratch = static_cast<uint32_t*>(addr);
    st.ctx.encode = reinterpret_cast<EncodeTiledFn>(fn);
    st.ctx.device = device;
    st.ctx.cfg.E = -1;                                   // forces the shape-dependent part below
    st.ready = true;
  }
  fb_ctx& ctx = st.ctx;
  if (memcmp(&ctx.cfg, cfg, sizeof(fb_config)) != 0) {
    // shape-dependent launch parameters (host arithmetic and function attributes only)
    const DeviceLimits limits = device_limits(device);
    if (!limits.usable) return FB_ERR_CUDA;
    ctx.cfg = *cfg;
    fb_status ss = setup_router_shape(&ctx, limits);
    if (ss == FB_OK) ss = set_up_device(&ctx, device, limits);
    if (ss != FB_OK) { ctx.cfg.E = -1; return ss; }
    ctx.split_mode = 0;                                  // the sums of an unsplit call, whatever the shape
    for (int i = 0; i < kMapCache; ++i) { ctx.x_maps[i] = MapEntry(); ctx.w_maps[i] = MapEntry(); }
  }
  ctx.counts_scratch = st.scratch;
  ctx.ticket = st.scratch + FB_STATIC_MAX_EXPERTS;
  ctx.status = status_word ? status_word : reinterpret_cast<int32_t*>(st.scratch + FB_STATIC_MAX_EXPERTS + 1);
  ctx.slice_counts = nullptr;                            // unused by the prediction pass
  if (T == 0)
    return cudaMemsetAsync(counts, 0, cfg->E * sizeof(uint32_t), stream) == cudaSuccess ? FB_OK : FB_ERR_CUDA;
  // The array keeps whatever the previous call (possibly one that was cut short) left in it.
  if (cudaMemsetAsync(st.scratch, 0, kStaticScratchWords * sizeof(uint32_t), stream) != cudaSuccess)
    return FB_ERR_CUDA;
  return launch_router(&ctx, router, x, T, fb::kModePredict, counts, topk_ids, nullptr, nullptr, nullptr, stream);
}
