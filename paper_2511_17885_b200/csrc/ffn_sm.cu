// Expert FFNs on the tcgen05 tensor cores, small-M form: the token rows are the MMA's N dimension.
//
// Section 3.1 makes the rows per expert small on purpose: a vision token activates K_v < K experts, so
// at batch 1 an expert sees a few dozen to ~120 rows (and a decode step a handful).  With the rows as
// the MMA's M dimension every k-step would pay a full 128-row instruction whatever the row count.  Here the roles are swapped:
//   D[128 output features, N token rows] (+)= W[128 features, 64] * X[N rows, 64]^T,   N = 16, 32, ... 128
// so that the tensor work of a tile and the activation box both shrink with the expert's rows, in steps
// of 16 and 32 rows.  One persistent kernel for both GEMMs: a warp that schedules tiles, one that feeds a TMA ring of four stages (six for a few tokens), one thread that issues
// the MMAs into two tensor-memory accumulator stages, four epilogue warps.  Tiles are handed out dynamically (an atomic counter), in
// an order that
//   - walks the routed tiles M-tile-major, so the rows of an M-tile are re-read from L2 by CTAs running at the same time while
//     every weight tile streams from HBM once,
//   - walks the shared-expert tiles N-block-major, so the CTAs running at the same time share one weight tile, and
//   - interleaves the two kinds evenly: routed tiles are bound by the weight stream and shared-expert tiles by the tensor pipe,
// all of GEMM-1's before GEMM-2's.  A GEMM-2 tile reads every feature of its M-tile's activations, so it waits until their count of
// arrivals is full; its weights are asked for meanwhile.  A tile belongs to a CTA only when that CTA claims it, so what a tile waits
// for is in the hands of a CTA that runs, whatever else holds SMs.
// Why one launch: as two, with the second's first weights asked for ahead, the SMs left GEMM-1 over 15-17 us (a tile is 1 MB of
// weights), and behind the last of them GEMM-2 waited 2 us for its start and 2 us for its first activations.  One token of
// the 64-expert layer 42.6 -> 40.7 us, 16 tokens of the 128-expert layer 133.4 -> 125.3, 200 tokens of the 64-expert layer 184.7 -> 177.0, 686 tokens
// of the 128-expert layer, pruned, 221.0 -> 208.6.  Where the call has other kernels to run meanwhile (the scores and the selection of a pruning
// stage), a few SMs are left to them (side_sms).
//   GEMM-1: a tile is (M-tile of one expert) x (128 intermediate features); two MMAs per k-step (gate
//           rows, up rows) share the activation operand; accumulators D_gate, D_up hold feature f in
//           TMEM lane f and token t in column t, so one thread owns gate and up of (f, t): SwiGLU in
//           registers, then act[row0 + t][f] with the warp's 32 lanes writing 32 neighbouring features.
//   GEMM-2: a tile is (M-tile) x (256 hidden features) as two MMAs (features 0-127, 128-255), or of 128
//           features with two k-blocks a stage where a call has too few tiles for the SMs; the
//           epilogue scales by the token's gate and adds the warp's 32 neighbouring features of one
//           token to the fp32 accumulator with one 128-byte reduction (or stores them, fixed-order mode).
// The transposed accumulator needs no shared-memory staging: for a fixed token the lanes of a warp already
// hold consecutive output features.
// When it runs: wherever CTA pairs do not (use_cta_pairs in internal.h).
// FP8 weight stream (WQ = 1): the expert matrices arrive as FP8 E4M3 bytes with one power-of-two scale per
// 128 x 128 block.  TMA brings the bytes (half the HBM traffic of bf16) into a ring of raw stages; eight more
// warps expand every weight box to bf16 in the 128-byte-swizzled layout the MMA reads (exactly: an E4M3 value
// has 4 significant bits and the scale is a power of two) into a second, two-deep ring; the activations stay
// bf16 and go from the raw stage straight to the MMA.  The contraction, the accumulators and the epilogues are
// those of the bf16 stream.
// Every wait is bounded; on expiry the CTA records FMMOE_ERR_TIMEOUT and leaves.
#include <cuda_bf16.h>

#include "internal.h"
#include "ptx.cuh"
#include "ffn_common.cuh"

namespace fmmoe {

constexpr int S_BK = 64;                              // one 128-byte swizzle atom of bf16
constexpr int S_FEW = 16, S_FEW_PAIRS = 96;            // a call of few tokens (FEW, below): up to so many, with up to so many pairs
constexpr int S_W_BYTES = 128 * S_BK * 2;             // one 128-feature weight box as bf16: 16 KB
constexpr int S_WQ_BYTES = 128 * S_BK;                // the same box as FP8 bytes: 8 KB
constexpr int S_THREADS = 224;                        // producer warp, issuer warp, four epilogue warps, tile-scheduler warp
constexpr int S_LOADERS = 128;                        // GEMM-1: four more warps that gather the routed rows of x
constexpr int S_CONVERTERS = 256;                     // FP8 stream: eight more warps that expand the weight boxes
constexpr int S_CVT_PIECES = 512 / S_CONVERTERS;      // 16-byte pieces of a weight box per converter thread
constexpr int S_TMEM_COLS = 512;                      // 2 accumulator stages x (2 x 128 columns)
// bf16 stream: a stage is [W0 16K][W1 16K][X].  FP8 stream: a raw stage is [W0 8K][W1 8K][X] and the
// expanded weights live in CVT_STAGES buffers of [W0 16K][W1 16K].
// FEW: calls of at most S_FEW tokens (a decode step), whose tiles have no more rows than the MMA's least N.  X needs 2 KB (4 KB with two
// k-blocks a stage) instead of 16, so that six stages fit, not four, and three expanded buffers, not two: 192 instead of 128 KB of weights on
// their way to an SM, which counts as long as the tiles do not keep the memory busy by themselves.  Four / six stages, us: 64 experts, top-6, two
// shared: 1 token 37.6 / 35.8, 2 45.6 / 44.6, 4 63.8 / 61.6, 16 (96 pairs) 116.1 / 115.4; 128 experts, top-8: 1 token 34.9 / 33.7, 8 94.3 /
// 93.3, 16 (128 pairs) 133.2 / 134.1; FP8: 1 token 47.5 / 46.8, 8 83.6 / 82.0, 16 tokens of 128 experts 112.9 / 113.8.
template <int WQ, int FEW> struct SmLayout {
  static constexpr int STAGES = FEW ? 6 : 4;
  static constexpr int CVT_STAGES = FEW ? 3 : 2;
  static constexpr int X_ROWS = FEW ? S_FEW : 128;
  static constexpr int X_BYTES = FEW ? 2 * S_FEW * S_BK * 2 : 128 * S_BK * 2;
  static constexpr int X2_OFF = X_BYTES / 2;          // two k-blocks a stage: where the second one's token rows lie
  static constexpr int W_RAW = WQ ? S_WQ_BYTES : S_W_BYTES;
  static constexpr int X_OFF = 2 * W_RAW;
  static constexpr int STAGE_BYTES = X_OFF + X_BYTES;
  static constexpr int CVT_OFF = STAGES * STAGE_BYTES;
  static constexpr int CVT_BYTES = WQ ? CVT_STAGES * 2 * S_W_BYTES : 0;
  static constexpr int BAR_OFF = CVT_OFF + CVT_BYTES;
  static constexpr int SMEM_BYTES = BAR_OFF + 1024 /*align*/ + 512 /*barriers, tile ring*/;
  static constexpr int BASE_THREADS = WQ ? S_THREADS + S_CONVERTERS : S_THREADS;
  static constexpr int THREADS = BASE_THREADS + S_LOADERS;
  // Registers: as for 512 threads where there are fewer, i.e. up to 128 a thread.  Left to itself the bf16 kernel takes 140; at 126
  // it spills nothing, and with what it leaves (20,480 registers) a window-score CTA of up to W = 5 or a small selection CTA fits beside it
  // (slowly: its loads queue behind the weight stream).  A pruned layer of 256 experts of 512 features, 6,500 tokens, W = 5: 423 -> 385 us; where
  // scoring is done in time on the SM that is left to it, no difference.
  static constexpr int BOUND = THREADS > 512 ? THREADS : 512;
};

__device__ __forceinline__ void red_add_f32(float* addr, float v) {
  asm volatile("red.global.add.f32 [%0], %1;" ::"l"(addr), "f"(v) : "memory");
}

// Token rows of a tile as the MMA sees them: a multiple of 16 (the instruction's N granularity for M = 128).
__device__ __forceinline__ int n_pad_of(int rows) { return rows <= 16 ? 16 : (rows + 15) & ~15; }

// Epilogues of up to N token rows of a 32-token block (a lane holds one feature): no work for columns that hold no row.  Stores
// under a condition for each of 32 columns in turn took 1,400 clocks for a single row.  With the gates asked for early and the
// first tile taken without the counter: 7 % off one token of the 64-expert layer, 1 % off 16 tokens of the 128-expert layer, 4 % off
// 200 tokens of the 64-expert one.
template <int N>
__device__ __forceinline__ void swiglu_rows(__nv_bfloat16* dst, int ld, const uint32_t (&g)[32], const uint32_t (&u)[32], int nt, int lane) {
  float a[N];
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const float g0 = __uint_as_float(g[j]);
    a[j] = __fdividef(g0, 1.f + __expf(-g0)) * __uint_as_float(u[j]);
  }
  store_rows_bf16<N>(dst, ld, a, nt, lane);
}
template <int N>
__device__ __forceinline__ void gated_rows(__nv_bfloat16* dst, int ld, float gate_l, const uint32_t (&v)[32], int nt, int lane) {
  float a[N];
#pragma unroll
  for (int j = 0; j < N; ++j) a[j] = __shfl_sync(0xffffffffu, gate_l, j) * __uint_as_float(v[j]);
  store_rows_bf16<N>(dst, ld, a, nt, lane);
}

// The kernel's tensor maps.
struct SmMaps {
  CUtensorMap x2[4];     // GEMM-2, routed: activations, boxes of 32, 64, 96 and 128 rows (FEW: 16)
  CUtensorMap xs[2];     // shared experts, [phase]: x, activations
  CUtensorMap w[2][3];   // [segment]: gate, up, down
};

template <int WQ, int FEW>
__global__ void __launch_bounds__((SmLayout<WQ, FEW>::BOUND), 1)
ffn_sm_kernel(const __grid_constant__ SmMaps maps, const GemmParams p) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  unsigned char* smem = smem_raw + ((1024 - (raw & 1023)) & 1023);   // 1024-byte aligned tiles (128B swizzle)
  using L = SmLayout<WQ, FEW>;
  constexpr int S_STAGES = L::STAGES, S_CVT_STAGES = L::CVT_STAGES, S_STAGE_BYTES = L::STAGE_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::BAR_OFF);
  uint64_t* full_bar = bars;                   // [S_STAGES]
  uint64_t* empty_bar = bars + S_STAGES;       // [S_STAGES]
  uint64_t* tfull_bar = bars + 2 * S_STAGES;   // [2]
  uint64_t* tempty_bar = tfull_bar + 2;        // [2]
  uint64_t* sfull_bar = tempty_bar + 2;        // [G_SCHED]
  uint64_t* sempty_bar = sfull_bar + G_SCHED;  // [G_SCHED]
  uint64_t* cfull_bar = sempty_bar + G_SCHED;  // [S_CVT_STAGES]  FP8 stream: expanded weights ready
  uint64_t* cempty_bar = cfull_bar + S_CVT_STAGES;   // [S_CVT_STAGES]
  volatile int* ring = reinterpret_cast<volatile int*>(cempty_bar + S_CVT_STAGES);   // [G_SCHED][G_SLOT_INTS]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(const_cast<int*>(ring) + G_SCHED * G_SLOT_INTS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* prod_half = abort_flag + 1;    // tiles the producer has taken half-way (paces the tile scheduler)

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint64_t budget = p.wait_budget_ns;

  if (threadIdx.x == 0) {
    // full: the producer and every loader thread, or the producer alone for all of them
    // a raw stage is free again once the MMAs have read its activations and (FP8 stream) every converter
    // warp has read its weight bytes (one arrival per warp: hundreds of per-thread arrivals on one barrier
    // would cost more than the conversion itself)
    for (int i = 0; i < S_STAGES; ++i) { mbar_init(&full_bar[i], 1 + S_LOADERS); mbar_init(&empty_bar[i], WQ ? 1 + S_CONVERTERS / 32 : 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&tfull_bar[i], 1); mbar_init(&tempty_bar[i], 128); }
    // readers of a tile: producer + issuer + 4 epilogue warps + the loader warps (+ the converter warps)
    for (int i = 0; i < G_SCHED; ++i) { mbar_init(&sfull_bar[i], 1); mbar_init(&sempty_bar[i], 6 + S_LOADERS / 32 + (WQ ? S_CONVERTERS / 32 : 0)); }
    for (int i = 0; i < S_CVT_STAGES; ++i) { mbar_init(&cfull_bar[i], S_CONVERTERS / 32); mbar_init(&cempty_bar[i], 1); }
    *abort_flag = 0;
    *prod_half = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, S_TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // Barriers, tensor memory and descriptors are set up.  A CTA whose first tile is one of a shared expert (the first p.shared_first are)
  // works on it while the router runs.  Whoever needs the router's record waits for it himself: the scheduler before the first
  // routed tile, the loaders before their first row, the epilogue before its first gate.  That this is safe hangs on where
  // the router lets its successor start: behind its own wait and behind its clearing of the counters, hence everything in front of the
  // layer (x, the weights, the last reader of this workspace) is done before this kernel starts.
  // One token of the 64-expert layer 43.8 -> 42.6 us, 200 tokens 185.8 -> 182.3.

  // the next tile from the ring, for one thread or a whole warp; false: no more (tile < 0) or a wait ran out (ok = false)
  auto wait_tile = [&](uint32_t it, TileInfo& ti, bool& ok, bool whole_warp) -> bool {
    const int slot = it % G_SCHED;
    const uint32_t sph = (it / G_SCHED) & 1;
    if (!(whole_warp ? mbar_wait_warp(&sfull_bar[slot], sph, abort_flag, budget) : mbar_wait(&sfull_bar[slot], sph, abort_flag, budget))) { ok = false; return false; }
    const int tile = ring[slot * G_SLOT_INTS];
    ti = slot_load(ring + slot * G_SLOT_INTS);
    if (whole_warp) __syncwarp();
    if (!whole_warp || lane == 0) mbar_arrive(&sempty_bar[slot]);
    return tile >= 0;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (elect_one()) {
      for (int i = 0; i < 4; ++i) tma_prefetch_desc(&maps.x2[i]);
      for (int i = 0; i < 3; ++i) tma_prefetch_desc(&maps.w[0][i]);
      if (p.shared_mtiles) { for (int i = 0; i < 2; ++i) tma_prefetch_desc(&maps.xs[i]); for (int i = 0; i < 3; ++i) tma_prefetch_desc(&maps.w[1][i]); }
      const uint64_t pol_stream = l2_policy_evict_first();
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      int issued = 0;        // k-blocks handed to the TMA engine so far
      bool stop = false;
      for (uint32_t it = 0; ok && !stop; ++it) {
        // the tile comes decoded from the scheduler warp: the producer touches no global memory but the TMA maps
        TileInfo ti;
        if (!wait_tile(it, ti, ok, false)) break;
        const Segment& sg = p.seg[ti.phase][ti.seg];
        const bool gemm2 = ti.phase != 0, fine = gemm2 && WQ == 0 && p.fine;
        // activation box: the smallest of 32 / 64 / 96 / 128 rows that covers the tile's (padded) rows
        const int bi = FEW ? 0 : ti.seg && !fine ? 3 : (n_pad_of(ti.rows) + 31) / 32 - 1;
        const CUtensorMap* mX = ti.seg ? &maps.xs[ti.phase] : &maps.x2[bi];
        const bool gather_x = !gemm2 && ti.seg == 0;   // the loader warps bring these rows
        const uint32_t x_bytes = gather_x ? 0u : FEW ? S_FEW * 128u : (uint32_t)(bi + 1) * 32u * 128u;
        const CUtensorMap* mW0 = &maps.w[ti.seg][gemm2 ? 2 : 0];
        const CUtensorMap* mW1 = &maps.w[ti.seg][gemm2 ? 2 : 1];
        // weights of a routed expert whose rows fit one M-tile are read exactly once: let them leave L2 first
        const bool stream_w = ti.seg == 0 && ti.single;
        const int x_row = ti.row0 + ti.group_local * sg.a_group_stride;
        const int w_y0 = ti.group_local * sg.b_rows_per_group + ti.nb * (!gemm2 || fine ? 128 : 256);
        const int w_y1 = gemm2 ? w_y0 + 128 : w_y0;
        const int k_all = sg.k_blocks, n_fill = fine ? (k_all + 1) >> 1 : k_all;
        const int kb_half = n_fill >> 1, hold = gemm2 ? -1 : p.test_withhold_stage;
        // a stage's bytes and its weights (the maps count columns in elements: bf16 elements, or FP8 bytes)
        auto load_w = [&](int st, int kb) {
          unsigned char* sW = smem + st * S_STAGE_BYTES;
          auto box = [&](unsigned char* dst, const CUtensorMap* m, int x, int y) {
            if (stream_w) tma_load_2d_hint(dst, m, &full_bar[st], x, y, pol_stream);
            else tma_load_2d(dst, m, &full_bar[st], x, y);
          };
          if (gemm2) mbar_arrive_n(&full_bar[st], S_LOADERS);      // the loaders have nothing to bring
          if (fine) {      // k-blocks 2 kb and 2 kb + 1 (the last stage of an odd count holds one)
            const int n = 2 * kb + 1 < k_all ? 2 : 1;
            mbar_arrive_expect_tx(&full_bar[st], (uint32_t)n * (L::W_RAW + x_bytes));
            for (int u = 0; u < n; ++u) box(sW + u * L::W_RAW, mW0, (2 * kb + u) * S_BK, w_y0);
          } else {
            mbar_arrive_expect_tx(&full_bar[st], 2u * L::W_RAW + x_bytes);
            box(sW, mW0, kb * S_BK, w_y0);
            box(sW + L::W_RAW, mW1, kb * S_BK, w_y1);
          }
        };
        // GEMM-2 on activations that are still being written: the weights of as many k-blocks as there are stages first
        int early = 0;
        if (gemm2) {
          if (!ti.ready) {
            int st = stage; uint32_t ph = phase;
            for (; early < S_STAGES && early < n_fill; ++early) {
              if (!mbar_wait(&empty_bar[st], ph ^ 1, abort_flag, budget)) { ok = false; break; }
              load_w(st, early);
              if (++st == S_STAGES) { st = 0; ph ^= 1; }
            }
            if (ok) ok = wait_rows(p, ti, abort_flag, budget);
            if (!ok) break;
          }
          fence_proxy_async_global();
        }
        for (int kb = 0; kb < n_fill; ++kb) {
          if (kb == kb_half) *prod_half = (int)it + 1;     // the scheduler may now claim the next tile
          if (kb >= early) {
            if (!mbar_wait(&empty_bar[stage], phase ^ 1, abort_flag, budget)) { ok = false; break; }
            if (issued == hold) {
              // Self-test hook (fmmoe_test_expire_wait): the producer stops here, before it has issued any copy
              // or arrival for this stage.  Nothing will ever complete the stage's barrier, so the issuer's
              // bounded wait runs out and the CTA leaves through its tear-down path.
              stop = true;
              break;
            }
            load_w(stage, kb);
          }
          ++issued;
          unsigned char* sX = smem + stage * S_STAGE_BYTES + L::X_OFF;
          if (fine) {
            for (int u = 0; u < (2 * kb + 1 < k_all ? 2 : 1); ++u) tma_load_2d(sX + u * L::X2_OFF, mX, &full_bar[stage], (2 * kb + u) * S_BK, x_row);
          } else if (!gather_x) {
            tma_load_2d(sX, mX, &full_bar[stage], kb * S_BK, x_row);
          }
          if (++stage == S_STAGES) { stage = 0; phase ^= 1; }
        }
      }
      if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
    }
  } else if (warp == 6) {
    // ------------------------------------------------------------ tile scheduler
    // Claims tiles from the global counter, decodes them (a global read of the M-tile list and a few
    // divisions) and publishes them through the slot ring: tile n+1 is claimed when the producer is half-way
    // through tile n.  Keeping this off the producer matters: its ring holds about as much work as a load takes
    // to arrive, so any pause of the producer starves the MMAs.
    if (elect_one()) {
      bool ok = true, waited = false;
      int n_mt_r = 0, n1 = 0, n_all = 0;
      for (uint32_t seq = 0; ok; ++seq) {
        if (seq >= 1) {
          const uint64_t t0 = global_timer_ns();
          while (*prod_half < (int)seq) {
            __nanosleep(64);
            if (*abort_flag || global_timer_ns() - t0 > budget) { ok = false; break; }
          }
          if (!ok) break;
        }
        const int id = atomicAdd(p.tile_counter, 1);
        if (id >= p.shared_first && !waited) {      // what is in front is done: the M-tile list can be read, the finalize pass may come
          pdl_wait();
          pdl_launch_dependents();
          waited = true;
          n_mt_r = routed_mtiles(p);
          n1 = p.phases & 1 ? phase_tiles(p, 0, n_mt_r) : 0;
          n_all = n1 + (p.phases & 2 ? phase_tiles(p, 1, n_mt_r) : 0);
        }
        const int tile = id < p.shared_first || id < n_all ? id : -1;
        TileInfo ti = {};
        if (tile >= 0) {
          const int ph = id >= p.shared_first && id >= n1;
          ti = decode_tile(p, ph, ph ? id - n1 : id, n_mt_r);
          if (ph) ti.ready = rows_ready(p, ti);
        }
        const int slot = seq % G_SCHED;
        const uint32_t sph = (seq / G_SCHED) & 1;
        if (!mbar_wait(&sempty_bar[slot], sph ^ 1, abort_flag, budget)) { ok = false; break; }
        slot_store(ring + slot * G_SLOT_INTS, tile, ti);
        mbar_arrive(&sfull_bar[slot]);
        if (tile < 0) break;
      }
      // a scheduler that gave up because another role aborted records nothing: the status word has the cause
      if (!ok && !*abort_flag) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ UMMA issuer
    if (elect_one()) {
      int stage = 0; uint32_t phase = 0;
      int as = 0; uint32_t aphase = 0;
      int cs = 0; uint32_t cphase = 0;
      bool ok = true;
      for (uint32_t it = 0; ok; ++it) {
        TileInfo ti;
        if (!wait_tile(it, ti, ok, false)) break;
        const uint32_t idesc = umma_idesc_bf16(128, n_pad_of(ti.rows));
        const bool gathered = ti.phase == 0 && ti.seg == 0, fine = ti.phase && WQ == 0 && p.fine;
        const int k_all = p.seg[ti.phase][ti.seg].k_blocks, k_blocks = fine ? (k_all + 1) >> 1 : k_all;
        if (!mbar_wait(&tempty_bar[as], aphase ^ 1, abort_flag, budget)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d0 = tmem_base + as * 256, d1 = d0 + 128;
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (!mbar_wait(&full_bar[stage], phase, abort_flag, budget)) { ok = false; break; }
          if (WQ && !mbar_wait(&cfull_bar[cs], cphase, abort_flag, budget)) { ok = false; break; }
          if (gathered) fence_proxy_async_smem();   // rows written by the loader warps' cp.async
          tc_fence_after();
          const uint32_t sS = smem_u32(smem + stage * S_STAGE_BYTES);
          const uint32_t sW = WQ ? smem_u32(smem + L::CVT_OFF + cs * 2 * S_W_BYTES) : sS;
          const uint64_t dw0 = umma_desc_sw128(sW);
          const uint64_t dw1 = umma_desc_sw128(sW + S_W_BYTES);
          const uint64_t dx = umma_desc_sw128(sS + L::X_OFF);
          if (fine) {
            const uint64_t dx1 = umma_desc_sw128(sS + L::X_OFF + L::X2_OFF);
#pragma unroll
            for (int k = 0; k < S_BK / 16; ++k) umma_bf16(d0, dw0 + 2 * k, dx + 2 * k, idesc, (kb | k) != 0);
            if (2 * kb + 1 < k_all) {
#pragma unroll
              for (int k = 0; k < S_BK / 16; ++k) umma_bf16(d0, dw1 + 2 * k, dx1 + 2 * k, idesc, true);
            }
          } else {
#pragma unroll
            for (int k = 0; k < S_BK / 16; ++k) {     // +32 bytes per K = 16 step inside the swizzle atom
              umma_bf16(d0, dw0 + 2 * k, dx + 2 * k, idesc, (kb | k) != 0);
              umma_bf16(d1, dw1 + 2 * k, dx + 2 * k, idesc, (kb | k) != 0);
            }
          }
          umma_commit(&empty_bar[stage]);   // stage reusable once these MMAs have read it
          if (++stage == S_STAGES) { stage = 0; phase ^= 1; }
          if (WQ) {
            umma_commit(&cempty_bar[cs]);   // and so is the buffer of expanded weights
            if (++cs == S_CVT_STAGES) { cs = 0; cphase ^= 1; }
          }
        }
        if (!ok) break;
        umma_commit(&tfull_bar[as]);        // both accumulators complete
        if (++as == 2) { as = 0; aphase ^= 1; }
      }
      if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
    }
  } else if (warp >= L::BASE_THREADS / 32) {
    // ------------------------------------------------------------ row loaders (GEMM-1, the last four warps)
    // Every stage of a routed tile: its rows x 128 bytes of x, row r = token row_token[row0 + r], written where a TMA box
    // with the 128-byte swizzle would put them (16-byte chunk c of row r at r*128 + ((c ^ (r & 7)) * 16)), so that no expert-ordered copy of x is written and read
    // back.  For GEMM-1's shared tiles the loaders only keep the stage barriers in step; GEMM-2's, which come last, do without them.
    const int lt = threadIdx.x - L::BASE_THREADS;      // 0..127
    const int chunk = lt & 7, rq = lt >> 3;            // eight lanes a row, rows rq, rq+16, ...
    const uint32_t dst0 = (uint32_t)(L::X_OFF + rq * 128 + ((chunk ^ (rq & 7)) << 4));
    int stage = 0; uint32_t phase = 0;
    bool ok = true, waited = false;
    const __nv_bfloat16* xg = p.x + chunk * 8;
    for (uint32_t it = 0; ok; ++it) {
      TileInfo ti;
      if (!wait_tile(it, ti, ok, true)) break;
      if (ti.phase) continue;
      const Segment& sg = p.seg[0][ti.seg];
      const bool gather_x = ti.seg == 0;
      if (gather_x && !waited) { pdl_wait(); waited = true; }      // row_token
      constexpr int ROUNDS = L::X_ROWS / 16;
      const __nv_bfloat16* src[ROUNDS];
#pragma unroll
      for (int i = 0; i < ROUNDS; ++i) {
        const int r = rq + 16 * i;
        src[i] = gather_x && r < ti.rows ? xg + (long long)p.row_token[ti.row0 + r] * p.ld_x : nullptr;
      }
      for (int kb = 0; kb < sg.k_blocks; ++kb) {
        if (!mbar_wait_warp(&empty_bar[stage], phase ^ 1, abort_flag, budget)) { ok = false; break; }
        if (gather_x) {
          const uint32_t sX = smem_u32(smem + stage * S_STAGE_BYTES) + dst0;
#pragma unroll
          for (int i = 0; i < ROUNDS; ++i)
            if (src[i]) cp_async_16(sX + i * 2048, src[i] + kb * S_BK);
          cp_async_arrive_noinc(&full_bar[stage]);
        } else {
          mbar_arrive(&full_bar[stage]);
        }
        if (++stage == S_STAGES) { stage = 0; phase ^= 1; }
      }
    }
    if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
  } else if (WQ && warp >= 7) {
    // ------------------------------------------------------------ weight converters (FP8 stream, warps 7..14)
    // Per k-block: two boxes of 128 rows x 64 FP8 bytes (row-major, 64-byte rows) -> two boxes of 128 rows x 64
    // bf16 in the 128-byte swizzle (16-byte chunk c of row r at r*128 + ((c ^ (r & 7)) * 16)).  A thread takes
    // 16 bytes (row p/4, bytes 16*(p%4) ..) at a time: one 16-byte load, two 16-byte stores; consecutive
    // threads read consecutive pieces and the eight lanes of a quarter-warp write eight different chunks.
    const int ct = threadIdx.x - S_THREADS;      // 0 .. S_CONVERTERS-1
    int stage = 0; uint32_t phase = 0;
    int cs = 0; uint32_t cphase = 0;
    bool ok = true;
    for (uint32_t it = 0; ok; ++it) {
      TileInfo ti;
      if (!wait_tile(it, ti, ok, true)) break;
      const Segment& sg = p.seg[ti.phase][ti.seg];
      // block scales of the tile's two weight boxes: lane l holds the exponent of 128-column block l of 32
      const int n_kb128 = (sg.k_blocks + 1) >> 1;
      const int rb0 = ti.phase ? 2 * ti.nb : ti.nb, rb1 = ti.phase ? 2 * ti.nb + 1 : ti.nb;
      const int rb_per_group = (sg.b_rows_per_group + 127) >> 7;
      const long long sc_base = (long long)ti.group_local * rb_per_group;
      const int8_t* sc0 = p.wscale[ti.phase][ti.seg][0];
      const int8_t* sc1 = p.wscale[ti.phase][ti.seg][1];
      int se0 = 0, se1 = 0;
      for (int kb = 0; kb < sg.k_blocks; ++kb) {
        if ((kb & 63) == 0 && (kb >> 1) + lane < n_kb128) {
          se0 = sc0[(sc_base + rb0) * n_kb128 + (kb >> 1) + lane];
          if (rb1 < rb_per_group) se1 = sc1[(sc_base + rb1) * n_kb128 + (kb >> 1) + lane];
        }
        // warp-uniform outcome: the arrivals below are made by one lane on behalf of the warp
        if (!__all_sync(0xffffffffu, mbar_wait(&full_bar[stage], phase, abort_flag, budget) &&
                                     mbar_wait(&cempty_bar[cs], cphase ^ 1, abort_flag, budget))) { ok = false; break; }
        const int e0 = __shfl_sync(0xffffffffu, se0, (kb >> 1) & 31), e1 = __shfl_sync(0xffffffffu, se1, (kb >> 1) & 31);
        const unsigned char* raw_w = smem + stage * S_STAGE_BYTES;
        unsigned char* out_w = smem + L::CVT_OFF + cs * 2 * S_W_BYTES;
#pragma unroll
        for (int box = 0; box < 2; ++box) {
          const uint32_t mbits = (uint32_t)(247 + (box ? e1 : e0)) << 7;      // bf16 2^(120 + scale exponent)
          const uint32_t m2 = mbits | (mbits << 16);
          const __nv_bfloat162 mul = *reinterpret_cast<const __nv_bfloat162*>(&m2);
          uint4 q[S_CVT_PIECES];
#pragma unroll
          for (int i = 0; i < S_CVT_PIECES; ++i)
            q[i] = *reinterpret_cast<const uint4*>(raw_w + box * S_WQ_BYTES + (i * S_CONVERTERS + ct) * 16);
#pragma unroll
          for (int i = 0; i < S_CVT_PIECES; ++i) {
            const int pce = i * S_CONVERTERS + ct, r = pce >> 2, c = pce & 3;
            uint32_t o[8];
            e4m3x4_to_bf16x4(q[i].x, mul, o[0], o[1]); e4m3x4_to_bf16x4(q[i].y, mul, o[2], o[3]);
            e4m3x4_to_bf16x4(q[i].z, mul, o[4], o[5]); e4m3x4_to_bf16x4(q[i].w, mul, o[6], o[7]);
            unsigned char* row = out_w + box * S_W_BYTES + r * 128;
            *reinterpret_cast<uint4*>(row + (((2 * c) ^ (r & 7)) << 4)) = make_uint4(o[0], o[1], o[2], o[3]);
            *reinterpret_cast<uint4*>(row + (((2 * c + 1) ^ (r & 7)) << 4)) = make_uint4(o[4], o[5], o[6], o[7]);
          }
        }
        fence_proxy_async_smem();            // the MMA reads these generic-proxy writes through the async proxy
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&cfull_bar[cs]);
          mbar_arrive(&empty_bar[stage]);    // this warp is done with the stage's weight bytes
        }
        if (++stage == S_STAGES) { stage = 0; phase ^= 1; }
        if (++cs == S_CVT_STAGES) { cs = 0; cphase ^= 1; }
      }
    }
    if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
  } else if (warp >= 2 && warp < 6) {
    // ------------------------------------------------------------ epilogue (warps 2..5)
    const int q = warp & 3;                 // TMEM lane quarter this warp may access = features 32q .. 32q+31
    int as = 0; uint32_t aphase = 0;
    bool ok = true, waited = false;
    for (uint32_t it = 0; ok; ++it) {
      TileInfo ti;
      if (!wait_tile(it, ti, ok, true)) break;
      const Segment& sg = p.seg[ti.phase][ti.seg];
      float gate[4];                        // GEMM-2: gates of the tile's rows, lane l: row 32 c + l; asked for before the accumulator is waited for
      if (ti.phase) {
        if (!waited) { pdl_wait(); waited = true; }      // row_gate, row_token
#pragma unroll
        for (int c = 0; c < 4; ++c)         // 1 in fixed-order mode: gates are applied by the ordered gather
          gate[c] = ti.seg == 0 && !p.deterministic && c * 32 + lane < ti.rows ? p.row_gate[ti.row0 + c * 32 + lane] : 1.f;
      }
      if (!mbar_wait_warp(&tfull_bar[as], aphase, abort_flag, budget)) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + as * 256 + (static_cast<uint32_t>(q * 32) << 16);
      const long long out_row0 = (long long)ti.row0 + (long long)ti.group_local * sg.out_group_stride;
      const int n_chunks = (ti.rows + 31) >> 5;
      if (ti.phase == 0) {
        const int feat0 = ti.nb * 128 + q * 32;
        const bool f_ok = feat0 < sg.n_valid;      // a multiple of 64: all 32 features or none
        __nv_bfloat16* dst = p.act[ti.seg] + out_row0 * sg.ld_out + feat0;
#pragma unroll 1
        for (int c = 0; c < n_chunks; ++c) {
          uint32_t g[32], u[32];
          tmem_ld32(taddr + c * 32, g);
          tmem_ld32(taddr + 128 + c * 32, u);
          tmem_ld_wait();
          const int nt = min(32, ti.rows - c * 32);      // warp-uniform
          if (f_ok) {
            __nv_bfloat16* d = dst + (long long)(c * 32) * sg.ld_out;
            if (nt <= 8) swiglu_rows<8>(d, sg.ld_out, g, u, nt, lane);
            else swiglu_rows<32>(d, sg.ld_out, g, u, nt, lane);
          }
        }
      } else {
        const bool fine = WQ == 0 && p.fine;       // one accumulator box, else two, 128 features apart
        const int feat_w = ti.nb * (fine ? 128 : 256) + q * 32;
#pragma unroll 1
        for (int c = 0; c < n_chunks; ++c) {
          const int nt = min(32, ti.rows - c * 32);      // warp-uniform
          const float gate_l = c < 2 ? (c ? gate[1] : gate[0]) : (c == 2 ? gate[2] : gate[3]);
          const int tok_l = p.pair || p.deterministic ? 0 : ti.seg ? ti.row0 + c * 32 + lane : lane < nt ? p.row_token[ti.row0 + c * 32 + lane] : 0;
#pragma unroll 1
          for (int box = 0; box < (fine ? 1 : 2); ++box) {
            const int feat0 = feat_w + box * 128;
            if (feat0 >= sg.n_valid) break;              // warp-uniform; a multiple of 64: all 32 features or none
            uint32_t v[32];
            tmem_ld32(taddr + box * 128 + c * 32, v);
            tmem_ld_wait();
            if (p.pair) {
              // pair-row mode: gate-scaled bf16 rows per pair; for one token the warp writes 64 contiguous bytes
              __nv_bfloat16* yp = p.yb[ti.seg] + (out_row0 + c * 32) * sg.ld_out + feat0;
              if (nt <= 8) gated_rows<8>(yp, sg.ld_out, gate_l, v, nt, lane);
              else gated_rows<32>(yp, sg.ld_out, gate_l, v, nt, lane);
            } else if (p.deterministic) {
              float* yb = p.y[ti.seg] + (out_row0 + c * 32) * sg.ld_out + feat0 + lane;
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (j < nt) yb[(long long)j * sg.ld_out] = __uint_as_float(v[j]);
            } else {
#pragma unroll
              for (int j = 0; j < 32; ++j) {
                const int tk = __shfl_sync(0xffffffffu, tok_l, j);
                const float gt = __shfl_sync(0xffffffffu, gate_l, j);
                if (j < nt) red_add_f32(p.acc + (long long)tk * sg.ld_out + feat0 + lane, gt * __uint_as_float(v[j]));   // the warp adds 128 contiguous bytes
              }
            }
          }
        }
      }
      tc_fence_before();
      mbar_arrive(&tempty_bar[as]);
      if (++as == 2) { as = 0; aphase ^= 1; }
      if (ti.phase == 0) publish_rows(p, ti, lane);
    }
    if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
  }

  // ---------------------------------------------------------------- teardown
  pdl_wait(); pdl_launch_dependents();      // long done, but for a scheduler that gave up: this grid ends behind the one in front
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) *(volatile int32_t*)p.gave_up = 1;      // what others wait for from here stays out
    // give copies still in flight time to land before the shared memory is released
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 200000ull) { }
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, S_TMEM_COLS);
  }
}

// ---------------------------------------------------------------- host side
// SMs that the GEMMs leave to the pruning stage of the same call.  Its window scores take one SM some 0.6 us a CTA up to W = 3, 1 us up to W = 5 and
// 5 us beyond, where two fit it and none beside a GEMM CTA; beside one the others take ten times as long.  They and selection (16 us)
// are to be through before the GEMMs are, which take at least as long as their weights' way from memory.  An SM more costs the GEMMs 0.2 %.
// Pruned layers, one SM / by this rule: 128 experts of 768, H 2,048, W = 8: 2,000 tokens 240 / 240 us (two), 2,800 270 / 256 (two), 3,400 287 /
// 270 (two); W = 5, 2,500 and 3,400 tokens: one, 247 and 270 (with two 247 and 271); 256 experts of 512, W = 8, 6,500 tokens 411 / 383 (three); short layers
// of 3,000 tokens, H 1,024, W = 3: 128 experts of 384 108 / 95 (five), 16 experts of 1,024 81 / 69 (five).
static int side_sms(const FfnArgs& a, int sm_count) {
  if (a.side_ctas == 0) return 0;
  const fmmoe_layer_desc& d = *a.d;
  const double pairs = (double)a.T * d.top_k, experts = pairs < d.n_experts ? pairs : d.n_experts;
  const double weights = 3.0 * d.hidden * (experts * d.inter + (double)d.n_shared * d.shared_inter) * (d.weight_format == FMMOE_WEIGHTS_FP8_BLOCK128 ? 1 : 2);
  const double scores_us = a.side_ctas * (a.side_window <= 3 ? 0.6 : a.side_window <= 5 ? 1.0 : 5.0), room_us = weights / 6.5e6 - 30.0;
  const double n = scores_us / (room_us > 16.0 ? room_us : 16.0);
  const int most = sm_count > 6 ? 6 : sm_count - 1;
  return n >= most ? most : (int)n + 1;
}

template <int WQ, int FEW>
static fmmoe_status launch_ffn_sm_impl(fmmoe_handle* h, const FfnArgs& a, cudaStream_t s) {
  using L = SmLayout<WQ, FEW>;
  const fmmoe_layer_desc& d = *a.d;
  const int H = d.hidden, I = d.inter, E = d.n_experts, Ns = d.n_shared, Is = d.shared_inter;
  if (!h->encode_tiled) return FMMOE_ERR_CUDA;
  if (a.T == 0) return FMMOE_OK;
  const int mtps = (int)((a.T + TC_BLOCK_M - 1) / TC_BLOCK_M);

  // GEMM-2 in tiles of 128 features (two k-blocks a stage keep the bytes in flight) where even those fit one round of the
  // SMs: a single token leaves 64 of 148 SMs with a 256-feature tile.  One token of the 64-expert layer (H 2,048, six
  // routed and two shared experts), when GEMM-2 was a launch of its own: GEMM-2 19.8 -> 16.7 us, the layer 51.0 -> 48.5 us.  In a second round the same
  // tiles would cost a second ramp-up.  Up to 32 rows, so that two activation boxes share the stage's room for one.
  const int64_t routed_rows = a.T * d.top_k;
  const int64_t mt_most = (routed_rows < E ? routed_rows : E) + (int64_t)Ns * mtps;
  const int sms = h->sm_count - side_sms(a, h->sm_count);
  const int fine = !WQ && a.T <= 32 && mt_most * ((H + 127) / 128) <= sms;
  const int nb2 = fine ? (H + 127) / 128 : (H + 255) / 256;

  SmMaps m;
  bool ok = true;
  for (int i = 0; i < 4; ++i) ok &= make_map(h, &m.x2[i], a.act, (uint64_t)a.p_max, I, FEW ? S_FEW : 32 * (i + 1));
  auto wmap = [&](CUtensorMap* map, const void* base, uint64_t rows, uint64_t cols) {
    return WQ ? make_map_u8(h, map, base, rows, cols, 128) : make_map(h, map, base, rows, cols, 128);
  };
  ok &= wmap(&m.w[0][0], a.w->w_gate, (uint64_t)E * I, H);
  ok &= wmap(&m.w[0][1], a.w->w_up, (uint64_t)E * I, H);
  ok &= wmap(&m.w[0][2], a.w->w_down, (uint64_t)E * H, I);
  if (Ns) {
    ok &= make_map(h, &m.xs[0], a.x, (uint64_t)a.T, H, L::X_ROWS);
    ok &= make_map(h, &m.xs[1], a.act_sh, (uint64_t)Ns * a.T, Is, fine && !FEW ? 32 : L::X_ROWS);
    ok &= wmap(&m.w[1][0], a.w->ws_gate, (uint64_t)Ns * Is, H);
    ok &= wmap(&m.w[1][1], a.w->ws_up, (uint64_t)Ns * Is, H);
    ok &= wmap(&m.w[1][2], a.w->ws_down, (uint64_t)Ns * H, Is);
  } else {      // never dereferenced without shared experts
    for (int i = 0; i < 2; ++i) m.xs[i] = m.x2[3];
    for (int i = 0; i < 3; ++i) m.w[1][i] = m.w[0][i];
  }
  if (!ok) return FMMOE_ERR_CUDA;

  GemmParams p = {};
  p.mtiles = a.mtiles; p.n_mtiles = a.n_mtiles; p.max_mtiles = a.max_mtiles;
  p.block_m = TC_BLOCK_M; p.shared_mtiles = Ns * mtps; p.mt_per_shared = mtps; p.T = a.T;
  p.done = a.done; p.gave_up = a.gave_up;
  p.seg[0][0] = Segment{(I + 127) / 128, H / S_BK, I, I, 0, 0, I};
  p.seg[0][1] = Segment{Ns ? (Is + 127) / 128 : 0, H / S_BK, Is, Is, 0, (int)a.T, Is};
  p.seg[1][0] = Segment{nb2, I / S_BK, H, H, 0, 0, H};
  p.seg[1][1] = Segment{Ns ? nb2 : 0, Ns ? Is / S_BK : 0, H, H, (int)a.T, (int)a.T, H};
  fill_params(p, a);
  p.wait_budget_ns = h->wait_budget_ns;
  p.fine = fine;

  bool& attr_set = h->sm_attr_set[WQ][FEW];
  if (!attr_set) {
    FMMOE_CUDA_TRY(cudaFuncSetAttribute(ffn_sm_kernel<WQ, FEW>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM_BYTES));
    attr_set = true;
  }
  const int grid = a.grid_override > 0 ? a.grid_override : sms;
  const int s_tiles = p.shared_mtiles * p.seg[0][1].n_nblocks;
  p.routed_first = grid;
  for (int ph = 1; ph <= 2; ++ph) {      // both at once, unless kernels are timed one by one
    if (ph == 2 && !h->profiling) break;
    p.phases = h->profiling ? ph : 3;
    p.shared_first = ph == 2 ? 0 : s_tiles < grid ? s_tiles : grid;
    p.tile_counter = a.tile_counters + (ph - 1);
    p.test_withhold_stage = ph == 1 ? a.test_withhold_stage : -1;
    { ProfScope ps(h, ph == 1 ? FMMOE_KERNEL_GEMM1 : FMMOE_KERNEL_GEMM2, s); FMMOE_CUDA_TRY(launch_pdl(ffn_sm_kernel<WQ, FEW>, dim3(grid), dim3(L::THREADS), L::SMEM_BYTES, s, 1, m, p)); }
    FMMOE_CUDA_TRY(cudaGetLastError());
    h->launches += 1;
  }
  return FMMOE_OK;
}

fmmoe_status launch_ffn_sm(fmmoe_handle* h, const FfnArgs& a, cudaStream_t s) {
  const bool few = a.T <= S_FEW && a.T * a.d->top_k <= S_FEW_PAIRS;
  if (a.d->weight_format == FMMOE_WEIGHTS_FP8_BLOCK128) return few ? launch_ffn_sm_impl<1, 1>(h, a, s) : launch_ffn_sm_impl<1, 0>(h, a, s);
  return few ? launch_ffn_sm_impl<0, 1>(h, a, s) : launch_ffn_sm_impl<0, 0>(h, a, s);
}

}  // namespace fmmoe
