// Internal declarations shared by the library's translation units (host side).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>
#include <stdio.h>

#include <utility>
#include <vector>

#include "../../include/fmmoe.h"

struct fmmoe_handle {
  int device;
  int sm_count;
  int max_smem_optin;
  int* d_status;        // device status word (0 = ok)
  int* h_status;        // pinned host mirror
  int64_t launches;     // kernels launched through this handle
  void* encode_tiled;   // cuTensorMapEncodeTiled entry point
  bool route_attr_set;  // dynamic shared memory opt-in done for the bf16 router
  bool sm_attr_set[2][2];   // ... for the small-M form of the expert GEMMs [FP8 weight stream][few tokens]
  bool tc2_attr_set;    // ... for the CTA-pair form
  bool tc2q_attr_set;   // ... and its FP8 weight stream
  bool f32_attr_set;    // ... for the fp32 expert GEMMs
  int64_t cta_pair_min_tokens;    // from this many tokens on the expert GEMMs run on CTA pairs (cta_group::2); -1: by use_cta_pairs
  int64_t pair_min_tokens;        // from this many tokens on the combine goes through per-pair bf16 rows (no atomics)
  int test_withhold_stage;        // self-test (fmmoe_test_expire_wait): armed for the next layer call, else -1
  uint64_t test_budget_ns;
  int test_route_cta, test_route_k_block;   // self-test (fmmoe_test_expire_route_wait): the CTA, armed for the next router it covers, else -1
  uint64_t test_route_budget_ns;
  uint32_t route_f32_attr_mask;   // ... for the fp32 router instantiations (bit = logits per lane; 0: the one for few experts)
  uint64_t wait_budget_ns;        // time budget of every bounded device-side wait
  // optional kernel timeline
  bool profiling;
  int prof_repeat;      // timeline on: launches of a short idempotent kernel issued back to back inside one event pair
  bool debug_sync;      // FMMOE_DEBUG_SYNC=1: synchronise after every kernel and report the first CUDA error on stderr
  int64_t debug_seq;    // kernels launched so far in debug mode
  std::vector<cudaEvent_t> ev_pool;
  size_t ev_used;
  struct ProfRec { int id; size_t start, stop; int reps; };
  std::vector<ProfRec> prof;
  // pipelined host I/O (created on first use): one stream per copy direction, a ring of events that
  // order them against the caller's compute stream, and a ring of events behind the host tickets
  static constexpr int kPipeEvents = 32, kTickets = 64;
  bool pipe_ready;
  cudaStream_t up_stream, down_stream;
  cudaEvent_t pipe_ev[kPipeEvents];
  uint64_t pipe_next;
  cudaEvent_t ticket_ev[kTickets];
  uint64_t ticket_next;
  // fmmoe_moe_forward_prune: the selection half of the pruning pass runs on a side stream
  bool side_ready;
  cudaStream_t side_stream;
  cudaEvent_t side_fork, side_join;
};

namespace fmmoe {

// Device-side status codes written to the status word (first writer wins).
enum : int { DEV_OK = 0, DEV_TIMEOUT = FMMOE_ERR_TIMEOUT, DEV_INTERNAL = FMMOE_ERR_INTERNAL };

constexpr int TC_BLOCK_M = 128;   // token rows per tile on the tensor-core path
constexpr int PAIR_BLOCK_M = 256; // token rows per tile of a CTA pair
constexpr int F32_BLOCK_M = 32;   // token rows per tile on the fp32 FMA path

// One M-tile of the expert-grouped row space.
struct MTile {
  int32_t group;  // expert id
  int32_t row0;   // first row (in the grouped order)
  int32_t rows;   // valid rows in this tile (1..block_m)
  int32_t pad;    // 1 if this is the only tile of its expert
};

// Rows per M-tile of an expert with `cnt` rows in `nt` = ceil(cnt / block_m) tiles.  Tiles of CTA pairs (block_m 256) share
// the rows evenly in steps of 32, the pair's granularity: 300 rows are 160 + 140, not 256 + 44 (whose second tile would
// read its weights for almost nothing).
__host__ __device__ static inline int mtile_rows(int cnt, int nt, int block_m) {
  if (block_m <= TC_BLOCK_M || nt == 0) return block_m;
  return ((cnt + nt - 1) / nt + 31) & ~31;
}

static inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Workspace layout of fmmoe_route / fmmoe_moe_forward (byte offsets).
struct WsPlan {
  size_t blk_cnt_off;           // int32 [E][ceil(T/32)] per-block expert counts / offsets (not cleared)
  size_t misc_off;              // int32 [misc_ints]: [0] number of routed M-tiles, [1],[2] tile counters of the expert GEMMs, [3] one of their CTAs gave up, from [8] on
                                // what has been written of each M-tile's activations (routed, then shared)
  int64_t misc_ints;
  size_t acc_off;               // fp32 [T,H] combine accumulator (atomic mode); the same region holds the bf16
                                // per-pair outputs [P_max + N_s*T, H] in pair-row mode (sized for the larger)
  size_t topk_idx_off, topk_w_off, inv_row_off;
  size_t expert_off_off, row_token_off, row_gate_off, mtiles_off;
  size_t act_off;               // dtype [P_max,I] SwiGLU activations
  size_t act_sh_off;            // dtype [N_s*T,I_s]
  size_t y_off;                 // fp32 [P_max,H]    (deterministic mode)
  size_t ysh_off;               // fp32 [N_s*T,H]    (deterministic mode)
  size_t total;
  int64_t p_max;
  int32_t max_mtiles;
};
bool plan_workspace(const fmmoe_layer_desc& d, int64_t T, uint32_t flags, WsPlan* p);

// Brackets one kernel launch with events when the handle's timeline is on.
// Kernels that give the same result when run twice in a row on the same arguments: with the timeline's repeat
// count above 1 their launch is issued that many times inside the event pair (`reps`), so that the launch
// latency an event pair adds to a 10-30 us kernel is amortised.  The scan / scatter pass works in place and
// the GEMMs consume a tile counter, so they always run once.
static inline bool prof_idempotent(int id) {
  return id == FMMOE_KERNEL_ROUTE || id == FMMOE_KERNEL_FINALIZE || id == FMMOE_KERNEL_PRUNE_INDEX ||
         id == FMMOE_KERNEL_PRUNE_SCORE || id == FMMOE_KERNEL_PRUNE_SELECT || id == FMMOE_KERNEL_PRUNE_COMPACT;
}
struct ProfScope {
  fmmoe_handle* h; cudaStream_t s; size_t rec; bool on; int kid; int reps;
  ProfScope(fmmoe_handle* h_, int id, cudaStream_t s_) : h(h_), s(s_), rec(0), on(h_->profiling), kid(id), reps(1) {
    if (!on) return;
    if (h->prof_repeat > 1 && prof_idempotent(id)) reps = h->prof_repeat;
    while (h->ev_pool.size() < h->ev_used + 2) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) { on = false; return; }
      h->ev_pool.push_back(e);
    }
    fmmoe_handle::ProfRec r{id, h->ev_used, h->ev_used + 1, reps};
    h->ev_used += 2;
    h->prof.push_back(r);
    rec = h->prof.size() - 1;
    cudaEventRecord(h->ev_pool[r.start], s);
  }
  ~ProfScope() {
    if (on) cudaEventRecord(h->ev_pool[h->prof[rec].stop], s);
    if (h->debug_sync) {
      ++h->debug_seq;
      cudaError_t e = cudaStreamSynchronize(s);
      if (e == cudaSuccess) e = cudaGetLastError();
      if (e != cudaSuccess) {
        fprintf(stderr, "fmmoe: kernel class %d (launch scope #%lld) failed: %s\n", kid, (long long)h->debug_seq, cudaGetErrorString(e));
        h->debug_sync = false;   // report the first failure only
      }
    }
  }
};

#define FMMOE_CUDA_TRY(expr)                         \
  do {                                               \
    cudaError_t _e = (expr);                         \
    if (_e != cudaSuccess) return FMMOE_ERR_CUDA;    \
  } while (0)

// Launch with programmatic dependent launch allowed (the kernel calls pdl_wait() before it touches
// data of earlier kernels), optionally as clusters of `cluster_x` CTAs.
template <typename... KArgs, typename... Args>
static inline cudaError_t launch_ex(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                    unsigned cluster_x, bool pdl, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n].val.programmaticStreamSerializationAllowed = 1;
    ++n;
  }
  if (cluster_x > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster_x; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
    ++n;
  }
  cfg.attrs = attr; cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
static inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                     unsigned cluster_x, Args&&... args) {
  return launch_ex(kernel, grid, block, smem, s, cluster_x, true, std::forward<Args>(args)...);
}

// ---- launchers (each returns after enqueueing; *launches is incremented per kernel) ----
struct RouteArgs {
  const void* x; const void* router_w; const float* router_b; const uint8_t* is_visual;
  int64_t T; int H, E, K, Kv; int reduce_on; int dtype;
  float* logits; float* probs; int32_t* topk_idx; float* topk_w; int32_t* inv_row;
  int32_t* blk_cnt;   // [E][route_blk_stride]: per token block (route_block_tokens) and expert, the number of selections
  float* acc_zero;    // [T,H] fp32 combine accumulator to clear (each CTA its own tokens' rows), or NULL
  int32_t* misc_zero;     // scheduler words, of which [1] to [misc_ints) are to be cleared, or NULL
  int64_t misc_ints;
  // the whole permutation in the router's kernel (route_fuses_permute): outputs as in PermuteArgs; inv_row is final
  int fuse; int block_m; int32_t* expert_off; int32_t* row_token; float* row_gate; MTile* mtiles; int32_t* n_mtiles;
};
// bf16 router: number of CTAs (a cluster) that share one 128-token tile by splitting the
// contraction.  Few tiles => split, so that more SMs stream X.
static inline int route_split(int64_t T, int H) {
  const int64_t tiles = (T + 127) / 128;
  const int kblocks = H / 64;
  if (tiles * 4 <= 160 && kblocks % 4 == 0) return 4;
  if (tiles * 2 <= 160 && kblocks % 2 == 0) return 2;
  return 1;
}
// Tokens per router CTA (= granularity of blk_cnt and of the in-block ranks the router leaves in inv_row).
static inline int route_block_tokens(int dtype, int64_t T, int H) {
  return dtype == FMMOE_BF16 ? 128 / route_split(T, H) : 32;
}
// Number of router CTAs = number of token blocks (the last tile's blocks may lie past T: they are empty).
static inline int route_num_blocks(int dtype, int64_t T, int H) {
  return dtype == FMMOE_BF16 ? (int)((T + 127) / 128) * route_split(T, H) : (int)((T + 31) / 32);
}
// Row pitch of the count table: a multiple of four, so that it can be read 16 bytes at a time.
static inline int route_blk_stride(int dtype, int64_t T, int H) { return (route_num_blocks(dtype, T, H) + 3) & ~3; }
// Batches whose router CTAs fit one (portable) cluster of eight: at most 256 tokens when the contraction is split over
// four CTAs.  They then see each other's selections in shared memory, and the two permutation kernels fall away
// (a layer of one token 58.3 -> 51.1 us, of sixteen 152 -> 144 us, together with the row gather in GEMM-1 that takes the
// place of the copy the scatter pass made at these sizes).  Beyond, clusters of sixteen are not portable.
static inline bool route_fuses_permute(int dtype, int64_t T, int H) { return route_num_blocks(dtype, T, H) <= 8; }
fmmoe_status launch_route(fmmoe_handle* h, const RouteArgs& a, cudaStream_t s);

struct PermuteArgs {
  const int32_t* topk_idx; const float* topk_w;
  int32_t* blk_cnt; int n_blk, ld_blk; int blk_tokens;   // router's block counts, row pitch ld_blk (scan: turned into offsets in place)
  int64_t T; int K, E; int block_m;
  int32_t* expert_off; int32_t* row_token; float* row_gate; int32_t* inv_row;
  MTile* mtiles; int32_t* n_mtiles;
};
fmmoe_status launch_permute(fmmoe_handle* h, const PermuteArgs& a, cudaStream_t s);

struct FfnArgs {   // both paths
  const fmmoe_layer_desc* d; const fmmoe_weights* w;
  const void* x; int64_t T; int64_t p_max;
  const MTile* mtiles; const int32_t* n_mtiles; int32_t max_mtiles;
  int32_t* tile_counters;   // [2] zeroed per call: tile schedulers of the expert GEMMs (of GEMM-1 and GEMM-2 launched one by one)
  int32_t* gave_up;         // small-M form, zeroed per call: a CTA has given up
  int32_t* done;            // small-M form, zeroed per call: arrivals per M-tile, routed ones, then (from max_mtiles on) shared ones
  int side_ctas, side_window;   // small-M form: window-score CTAs of this call's pruning stage, which run beside the expert GEMMs (0: none), and their W
  const int32_t* row_token; const float* row_gate;
  void* act; void* act_sh;
  float* acc;            // atomic mode
  float* y; float* ysh;  // deterministic mode
  void* yb; void* ybsh;  // pair-row mode (bf16)
  int deterministic;
  int pair;              // GEMM-2 stores gate-scaled bf16 rows per pair; the finalize pass sums them per token
  int* d_status;
  int test_withhold_stage;   // bf16, self-test only (-1: off)
  int grid_override;         // bf16, self-test only: CTAs or CTA pairs to launch (0: one per SM)
};
fmmoe_status launch_ffn_sm(fmmoe_handle* h, const FfnArgs& a, cudaStream_t s);    // bf16, tcgen05, token rows as N (gathers its rows of x)
fmmoe_status launch_ffn_tc2(fmmoe_handle* h, const FfnArgs& a, cudaStream_t s);   // bf16, tcgen05, CTA pairs, token rows as N, 256-row tiles
// Which form a bf16 layer takes.  What pairs save grows with the rows of an expert (weights are read once per 256 rows, not per 128, and the
// operands' way into an SM is shorter); the small-M form saves a launch in plain stream order, GEMM-1's tail and, below 128 rows, nothing
// by reading weights twice.
// Where the host knows how many tokens are vision tokens (a call with a pruning stage, a stack: `n_vis`), the line is drawn in rows that
// exist, shared experts among them (each has a row per token, which is what pairs are good at): an average of 116, 104 with FP8 weights.
// Small-M / pairs, us a layer in a sustained loop, average rows in brackets.  bf16, 128 experts, top-8, no shared: 2,048 tokens
// mostly vision (69) 221 / 233, 3,000 (100) 247 / 254, 3,584 with its stage (120) 290 / 271, 4,300 (144) 316 / 292; text 1,536 (96) 234 / 249, 1,792
// (112) 246 / 259, 2,048 (128) 284 / 270.  64 experts, top-6, two shared: text 1,024 (124) 256 / 250, 1,400 (170) 301 / 288; mostly vision 2,048
// (162) 288 / 283, 3,000 (237) 360 / 347.  FP8, with the stage, mostly vision, 128 experts: 2,400 (80) 272 / 281, 2,700 (90) 282 / 287, 2,850 (95) 294 / 290,
// 3,000 (100) 313 / 312, 3,150 (105) 320 / 314, 3,300 (110) 327 / 322, 3,584 (120) 336 / 330; 64 experts: 1,024 (81) 250 / 257, 1,200 (95) 270 / 263, 1,400
// (111) 292 / 287, 2,048 (162) 356 / 335; text, 128 experts: 1,792 (112) 261 / 284, 1,920 (120) 289 / 288, 2,048 (128) 316 / 292.  (While the power cap does
// not bite, in bursts, FP8 crosses later: 3,150 tokens 300 / 306, 3,450 317 / 318, 3,584 324 / 321; 64 experts 1,400 275 / 278, 1,550 299 / 293.)
// Where only the device knows, every token counts with top_k and shared experts do not: from 128 rows, 160 with FP8 weights.  Text-only calls
// cross there; mostly vision, which has half the rows counted, goes to pairs too early (5 % at 2,048 tokens of the 128-expert layer).
// And only where pairs have a tile for every SM.  That side is drawn too wide: small-M / pairs on text, 32 experts of 512 features,
// top-4: 512 tokens (64 rows) 56 / 64, 1,024 tokens (128 rows, 128 tiles) 73 / 66, 2,048 94 / 91; 64 experts of 256 features: 2,048
// tokens (128 rows, 128 tiles) 85 / 76, 4,096 115 / 113.
constexpr int64_t kCtaPairRows = 116, kCtaPairRowsFp8 = 104, kCtaPairTopK = 128, kCtaPairTopKFp8 = 160, kCtaPairMinTokens = 256;
// n_vis: vision tokens among the T, or -1; reduce_on: they take K_v experts.
static inline bool use_cta_pairs(const fmmoe_handle* h, const fmmoe_layer_desc& d, int64_t T, int64_t n_vis = -1, bool reduce_on = false) {
  if (d.dtype != FMMOE_BF16) return false;
  if (h->cta_pair_min_tokens >= 0) return T >= h->cta_pair_min_tokens;
  const bool fp8 = d.weight_format == FMMOE_WEIGHTS_FP8_BLOCK128, known = n_vis >= 0;
  const int64_t pairs = known && reduce_on ? (T - n_vis) * d.top_k + n_vis * d.top_k_vis : T * d.top_k;
  const bool enough = known ? pairs + d.n_shared * T >= (fp8 ? kCtaPairRowsFp8 : kCtaPairRows) * ((int64_t)d.n_experts + d.n_shared)
                            : pairs >= (fp8 ? kCtaPairTopKFp8 : kCtaPairTopK) * d.n_experts;
  const int64_t mtiles = pairs / PAIR_BLOCK_M > d.n_experts ? pairs / PAIR_BLOCK_M : d.n_experts;
  return T >= kCtaPairMinTokens && enough && mtiles * ((d.inter + 127) / 128) >= h->sm_count;
}
// Combine: every pair's gate-scaled row is written once in bf16 and summed per token in a fixed order
// (no atomics, reproducible bit for bit).  Measured against the atomic fp32 accumulator it is equal below
// 512 tokens and 2-4 % of a step faster from there on (the accumulator, T*H*4 bytes, stops fitting the L2
// cache next to the activations around 8,192 tokens and then pages through HBM), so it is the default at
// every size; FMMOE_PAIR_ROWS_MIN_TOKENS=n keeps the atomic combine below n tokens.
constexpr int64_t kPairMinTokensDefault = 0;
static inline bool use_pair_rows(const fmmoe_handle* h, const fmmoe_layer_desc& d, int64_t T, uint32_t flags) {
  return d.dtype == FMMOE_BF16 && !(flags & FMMOE_FLAG_DETERMINISTIC) && T >= h->pair_min_tokens;
}
fmmoe_status launch_ffn_f32(fmmoe_handle* h, const FfnArgs& a, cudaStream_t s);   // fp32 FMA

// One launch's sequences of a pruning stage.
struct PruneSeqs {
  static constexpr int MAX = FMMOE_MAX_SEQS_PER_LAUNCH;
  int n_seq;
  int n_vis[MAX], m[MAX], d[MAX];
  int win_off[MAX + 1];          // first window of each sequence in this launch
  long long seq_off[MAX + 1];    // token offsets
  long long out_off[MAX + 1];    // output row offsets
};
// A pruning stage whose rows the finalize pass writes itself (fmmoe_moe_forward_prune): what selection left for it.
struct FinalizePrune {
  const int32_t* pos;        // [T] output row of a copied token, -1 for others
  void* x_out;
  const int2* merges;        // per sequence, from win_off: (output row, rank of the first member) of each merged window
  const int32_t* vis_list;   // [T] token of a sequence's v-th vision token at seq_off + v
  int W, merge_mode, n_merges;
  PruneSeqs sq;
};

struct FinalizeArgs {
  const void* x; void* out; int64_t T; int H, K, n_shared; int dtype; int add_residual; int deterministic;
  const float* acc; const float* y; const float* ysh; const int32_t* inv_row; const float* topk_w;
  int pair; const void* yb; const void* ybsh;   // pair-row mode: bf16 [P,H] gate-scaled rows, [N_s*T,H] shared rows
  const FinalizePrune* prune;                   // pair-row mode, rows of up to 4 KB: also write the pruned rows (or NULL)
};
fmmoe_status launch_finalize(fmmoe_handle* h, const FinalizeArgs& a, cudaStream_t s);

// fmmoe_moe_forward for a caller that knows how many of its T tokens are vision tokens.
fmmoe_status moe_forward_vis(fmmoe_handle* h, const fmmoe_layer_desc* d, const fmmoe_weights* w, const void* x, const uint8_t* is_visual,
                             int64_t T, int64_t n_vis, uint32_t flags, void* out, const fmmoe_route_out* route, void* workspace,
                             size_t workspace_bytes, void* cuda_stream);

constexpr int SC_WIN = 8;      // windows that a CTA of the window scores takes
// start-up work of the pruning pass (module load, scratch address, shared-memory opt-in); device current
fmmoe_status prune_prepare(fmmoe_handle* h);

// Whether an output that selection writes lies over the mask it reads (a caller may compact the mask in place): then the
// gather pass writes these outputs, and no `fused` form is used.
bool prune_outputs_over_mask(const uint8_t* is_visual, int64_t T, int64_t T_out, const uint8_t* is_visual_out,
                             const int32_t* keep_idx, const uint8_t* kind);

// fmmoe_prune_visual in two phases (bit 0: ranks, scores, selection on s_select; bit 1: rows on s_rows).  With `fused`
// (at most FMMOE_MAX_SEQS_PER_LAUNCH sequences) selection leaves the inverse map for the finalize pass, which takes the place of phase 2.
fmmoe_status prune_visual_phases(fmmoe_handle* h, const fmmoe_prune_params* p, const float* probs, int32_t n_experts,
                                 const float* attn, const void* x, int32_t dtype, int32_t hidden,
                                 const uint8_t* is_visual, const int64_t* seq_off, const int64_t* n_vis,
                                 const int64_t* n_retain, int32_t n_seq, void* x_out, uint8_t* is_visual_out,
                                 int32_t* keep_idx, uint8_t* kind, int64_t* out_seq_off, void* workspace,
                                 size_t workspace_bytes, int phases, cudaStream_t s_select, cudaStream_t s_rows,
                                 FinalizePrune* fused = nullptr);

}  // namespace fmmoe
