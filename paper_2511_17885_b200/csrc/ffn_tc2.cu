// Expert FFNs on the tcgen05 tensor cores with CTA pairs (cta_group::2), the token rows as the MMA's N dimension.
//
//   D[256 weight rows, N token rows] (+)= W[256, 64] * X[N, 64]^T,   N = 32, 64, ... 256
// A tile is (token tile of one expert: up to 256 of its rows) x (256 weight rows).  The pair shares one MMA of M = 256:
//   cluster rank r (0 = leader, 1 = partner):
//     W   GEMM-1: 64 gate rows and the 64 up rows of the same features (128 features a tile, 64 a CTA); GEMM-2: 128 rows of
//         W_down (256 hidden features a tile)                                       16 KB per 64-deep k-block, own TMA loads
//     X   rows r * N/2 .. of the token tile                                         up to 16 KB, read by both CTAs' MMAs
//     D   the CTA's 128 weight rows x all N tokens, in its own tensor memory (lane = weight row, column = token)
// Why: one CTA with 256 weight rows and 128 token rows a tile takes 48 KB into its SM per k-block and 512 clocks of tensor work
// (96 B/clk) and reads an expert's weights once per 128 rows.  Here it is 32 KB and once per 256 rows, in steps of 32 (an expert of
// 480 rows is two tiles of 240), and the operand reads of the MMAs fall from 96-128 to 64 B/clk as well.
// What bounds it (clocks inside the kernel, one launch): with about 100 rows an expert both GEMMs stream the weights at
// 6.2-6.5 TB/s (658-724 clocks a k-block); with 200 or more the tensor pipe (485-500 clocks a k-block of 207-240 rows, 414-480
// of MMAs); in a sustained loop the 1 kW cap on top (1,230 and 1,030 MHz on 14,336 tokens of the 128-expert layer and 19,456 of the
// 64-expert one).  GEMM-1 / GEMM-2 by themselves (single launches under the profiler, 1.5-1.7 GHz), against one CTA a tile with the
// token rows as M: 14,336 tokens 338 -> 279 / 185 -> 153 us, 3,584 tokens 153 -> 133 / 82 -> 72, 2,432 tokens 163 -> 154 / 93 -> 85.
//   Roles per CTA: warp 0 TMA producer; warp 1 MMA issuer (leader) or relay (partner, GEMM-1: passes "my loaders' rows of this
//   stage have landed" on to the leader); warps 2-5 and four more epilogue; warp 6 tile scheduler; GEMM-1: four loader warps
//   that gather the routed rows of x by token with cp.async into the 128-byte-swizzled layout; FP8 stream: eight converter warps
//   and a producer for the rows.
//   Every role that waits on a ring also arrives in it, once a stage: a wait by parity tells a phase from the one before, not from
//   the one before that.
//   Barriers: the partner's TMA loads credit their bytes to the LEADER's full barrier; the leader's commit arrives on both
//   CTAs' empty / accumulator-full barriers (multicast commit: no data is multicast anywhere); the partner's epilogue warps
//   arrive on the leader's accumulator-empty barrier through the cluster.
//   GEMM-1's epilogue: gate rows sit in lanes 0-63, the up rows of the same features in lanes 64-127, so the warps q and q + 2
//   swap halves of every 32-token block through shared memory: each then owns 16 tokens x 32 features, gate and up.
// FP8 weight stream (WQ = 1, the format of ffn_sm.cu): every CTA expands its own 128 weight rows once per 256 token rows, where the
// small-M form expands 256 rows per 128: a layer of 3,584 tokens and 128 experts takes 12 % less time than in that form.
// Every wait on a barrier is bounded; on expiry the CTA records FMMOE_ERR_TIMEOUT and leaves (its partner's waits then run out
// too), and both still meet at the cluster barrier of the tear-down.
// The kernels are launched in plain stream order: launched with programmatic dependent launch, a run of a few hundred steps
// stalled in one of the hardware waits that cannot be bounded (cluster barrier, pair allocation, grid dependency).
#include <cuda_bf16.h>

#include "internal.h"
#include "ptx.cuh"
#include "ffn_common.cuh"

namespace fmmoe {

constexpr int P_BK = 64;
constexpr int P_W_BYTES = 128 * P_BK * 2;          // 16 KB: this CTA's half of the weight tile
constexpr int P_X_ROWS = PAIR_BLOCK_M / 2;         // room for this CTA's half of the token tile
constexpr int P_X_BYTES = P_X_ROWS * P_BK * 2;     // 16 KB
// epilogue, per warp: GEMM-1 [2 buffers][32 lanes][16 tokens] fp32 swapped with another warp; GEMM-2 32 gates
constexpr int P_XCH_BYTES = 8 * 2 * 16 * 32 * 4;
constexpr int P_BASE_THREADS = 224;                // producer, issuer, four epilogue warps, tile scheduler
constexpr int P_LOADERS = 128;
constexpr int P_CONVERTERS = 256;                  // FP8 stream: two groups of four warps that take alternate k-blocks
constexpr int P_TMEM_COLS = 512;
// bf16 stream: a stage is [W 16K][X 16K].  FP8 stream: the weight bytes, the token rows and the expanded weights have a ring
// each: a weight box is 8 KB, so that ten of them are in flight (with five, bound to the stages of the token rows, 512 tokens
// of the 128-expert layer took 243 us).
template <int WQ> struct PairLayout {
  static constexpr int W_RAW = WQ ? P_W_BYTES / 2 : P_W_BYTES;
  static constexpr int W_STAGES = WQ ? 10 : 6;
  static constexpr int X_STAGES = WQ ? 4 : 6;
  static constexpr int W_PITCH = WQ ? W_RAW : W_RAW + P_X_BYTES;
  static constexpr int X_OFF = WQ ? W_STAGES * W_RAW : W_RAW;
  static constexpr int X_PITCH = WQ ? P_X_BYTES : W_PITCH;
  static constexpr int CVT_OFF = WQ ? X_OFF + X_STAGES * P_X_BYTES : 0;
  static constexpr int CVT_STAGES = 3;
  static constexpr int XCH_OFF = WQ ? CVT_OFF + CVT_STAGES * P_W_BYTES : W_STAGES * W_PITCH;
  static constexpr int BAR_OFF = XCH_OFF + P_XCH_BYTES;
  static constexpr int SMEM_BYTES = BAR_OFF + 1024 /*align*/ + 1024 /*barriers, tile rings*/;
};
template <int MODE, int WQ> constexpr int pair_threads() {      // loaders, four more epilogue warps, converters and the rows' producer
  return P_BASE_THREADS + (MODE == 0 ? P_LOADERS : 0) + 128 + (WQ ? P_CONVERTERS + 32 : 0);
}

// Token rows of a tile as the MMA sees them: a multiple of 32 (each CTA supplies half, in steps of 16).
__device__ __forceinline__ int pair_n_pad(int rows) { return (rows + 31) & ~31; }

template <int MODE, int WQ>
__global__ void __launch_bounds__((pair_threads<MODE, WQ>()), 1)
ffn_tc2_kernel(const __grid_constant__ CUtensorMap tmX32, const __grid_constant__ CUtensorMap tmX64,
               const __grid_constant__ CUtensorMap tmX96, const __grid_constant__ CUtensorMap tmX128,
               const __grid_constant__ CUtensorMap tmXs,
               const __grid_constant__ CUtensorMap tmW0_r, const __grid_constant__ CUtensorMap tmW1_r,
               const __grid_constant__ CUtensorMap tmW0_s, const __grid_constant__ CUtensorMap tmW1_s,
               const GemmParams p) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  unsigned char* smem = smem_raw + ((1024 - (raw & 1023)) & 1023);   // the same offset in both CTAs of the pair
  using L = PairLayout<WQ>;
  float* xch = reinterpret_cast<float*>(smem + L::XCH_OFF);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::BAR_OFF);
  uint64_t* full_bar = bars;                          // [X_STAGES]  used in the leader: both CTAs' bytes of a stage
  uint64_t* empty_bar = full_bar + L::X_STAGES;       // [X_STAGES]  per CTA: the MMAs have read this CTA's stage
  uint64_t* xfull_bar = empty_bar + L::X_STAGES;      // [X_STAGES]  used in the partner (GEMM-1): its loaders' rows have landed
  uint64_t* wfull_bar = xfull_bar + L::X_STAGES;      // [W_STAGES]  per CTA, FP8 stream: this CTA's weight bytes have landed
  uint64_t* wempty_bar = wfull_bar + L::W_STAGES;     // [W_STAGES]  per CTA, FP8 stream: its converters have read them
  uint64_t* cfull_bar = wempty_bar + L::W_STAGES;     // [CVT_STAGES] used in the leader, FP8 stream: both CTAs' weights are expanded
  uint64_t* cempty_bar = cfull_bar + L::CVT_STAGES;   // [CVT_STAGES] per CTA, FP8 stream: the MMAs have read them
  uint64_t* tfull_bar = cempty_bar + L::CVT_STAGES;   // [2]             per CTA: accumulator stage complete
  uint64_t* tempty_bar = tfull_bar + 2;            // [2]             used in the leader: both CTAs' epilogues have drained it
  uint64_t* xch_bar = tempty_bar + 2;              // [4 warp pairs][2 buffers]
  uint64_t* sfull_bar = xch_bar + 8;               // [G_SCHED]       per CTA: a tile is in this CTA's ring
  uint64_t* sempty_bar = sfull_bar + G_SCHED;      // [G_SCHED]       per CTA: every reader has read it
  uint64_t* mfull_bar = sempty_bar + G_SCHED;      // [G_SCHED]       used in the partner: a tile from the leader is in its mailbox
  uint64_t* mempty_bar = mfull_bar + G_SCHED;      // [G_SCHED]       used in the leader: the partner has taken it out
  volatile int* ring = reinterpret_cast<volatile int*>(mempty_bar + G_SCHED);   // [G_SCHED][G_SLOT_INTS]
  volatile int* mailbox = ring + G_SCHED * G_SLOT_INTS;                         // [G_SCHED][G_SLOT_INTS]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(const_cast<int*>(mailbox) + G_SCHED * G_SLOT_INTS);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* prod_pace = abort_flag + 1;        // leader: tiles after which the scheduler may claim one more (set by its producer)
  volatile int* done = abort_flag + 2;             // [2] k-blocks and tiles this CTA took part in (p.check_drained)

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();         // 0: leader, 1: partner
  const bool leader = rank == 0;
  const uint64_t budget = p.wait_budget_ns;

  if (threadIdx.x == 0) {
    // full: the leader's producer (+ every loader thread of the leader + the partner's relay); xfull: the partner's loader threads and, in
    // the FP8 stream, its producer of the rows
    for (int i = 0; i < L::X_STAGES; ++i) {
      mbar_init(&full_bar[i], MODE == 0 ? 1 + P_LOADERS + 1 : 1);
      mbar_init(&empty_bar[i], 1);
      mbar_init(&xfull_bar[i], P_LOADERS + (WQ ? 1 : 0));
    }
    for (int i = 0; WQ && i < L::W_STAGES; ++i) { mbar_init(&wfull_bar[i], 1); mbar_init(&wempty_bar[i], P_CONVERTERS / 64); }
    // accumulator-empty: one arrival per epilogue warp of both CTAs
    for (int i = 0; i < 2; ++i) { mbar_init(&tfull_bar[i], 1); mbar_init(&tempty_bar[i], 16); }
    for (int i = 0; i < 8; ++i) mbar_init(&xch_bar[i], 2);
    for (int i = 0; i < L::CVT_STAGES; ++i) { mbar_init(&cfull_bar[i], 2 * (P_CONVERTERS / 64)); mbar_init(&cempty_bar[i], 1); }
    // readers of a tile: producer, issuer or relay (the partner has none in GEMM-2), eight epilogue warps, in GEMM-1 four loader
    // warps, in the FP8 stream eight converter warps and the rows' producer
    for (int i = 0; i < G_SCHED; ++i) {
      mbar_init(&sfull_bar[i], 1); mbar_init(&sempty_bar[i], (MODE == 0 ? 14 : leader ? 10 : 9) + (WQ ? P_CONVERTERS / 32 + 1 : 0));
      mbar_init(&mfull_bar[i], 1); mbar_init(&mempty_bar[i], 1);
    }
    *abort_flag = 0;
    *prod_pace = 0;
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, P_TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  cluster_arrive();
  const uint32_t tmem_base = *tmem_slot;

  pdl_wait();
  const int n_mt_r = routed_mtiles(p);
  cluster_wait();              // the partner's barriers exist before anything of this CTA can signal them
  const int total_tiles = phase_tiles(p, MODE, n_mt_r);

  // the next tile from this CTA's ring, for one thread or a whole warp; false: no more (tile < 0) or a wait ran out (ok = false)
  auto wait_tile = [&](uint32_t it, TileInfo& ti, bool& ok, bool whole_warp = false) -> bool {
    const int slot = it % G_SCHED;
    const uint32_t sph = (it / G_SCHED) & 1;
    if (!(whole_warp ? mbar_wait_warp(&sfull_bar[slot], sph, abort_flag, budget) : mbar_wait(&sfull_bar[slot], sph, abort_flag, budget))) { ok = false; return false; }
    const int tile = ring[slot * G_SLOT_INTS];
    ti = slot_load(ring + slot * G_SLOT_INTS);
    return tile >= 0;
  };
  auto release_tile = [&](uint32_t it) { mbar_arrive(&sempty_bar[it % G_SCHED]); };      // one thread per reader

  if (warp == 0 || (WQ && warp == pair_threads<MODE, WQ>() / 32 - 1)) {
    // ------------------------------------------------------------ TMA producers (both CTAs)
    // One thread for a stage of weights and rows; in the FP8 stream one for the weight bytes (warp 0) and one for the rows (the
    // last warp), each at the pace of its own ring.
    const bool weights = warp == 0, rows = !WQ || warp != 0;
    if (elect_one()) {
      if (MODE == 1 && rows) { tma_prefetch_desc(&tmX32); tma_prefetch_desc(&tmX64); tma_prefetch_desc(&tmX96); tma_prefetch_desc(&tmX128); }
      if (weights) { tma_prefetch_desc(&tmW0_r); if (MODE == 0) tma_prefetch_desc(&tmW1_r); }
      if (p.shared_mtiles) { if (rows) tma_prefetch_desc(&tmXs); if (weights) { tma_prefetch_desc(&tmW0_s); tma_prefetch_desc(&tmW1_s); } }
      const uint32_t full_leader = cluster_map_shared(smem_u32(full_bar), 0);   // the leader's full barriers
      const int n_stages = weights ? L::W_STAGES : L::X_STAGES;
      const uint64_t pol_stream = l2_policy_evict_first();
      uint64_t* free_bar = WQ && weights ? wempty_bar : empty_bar;
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      int n_kb = 0, issued = 0;      // k-blocks of the tiles taken; asked for
      bool stop = false;
      uint32_t it = 0;
      for (; ok && !stop; ++it) {
        TileInfo ti;
        if (!wait_tile(it, ti, ok)) break;
        release_tile(it);
        const Segment& sg = p.seg[MODE][ti.seg];
        n_kb += sg.k_blocks;
        const int half = pair_n_pad(ti.rows) >> 1;
        // token rows by TMA: the smallest box of 32 / 64 / 96 / 128 rows that covers the half (shared experts: all the room)
        const int bi = (half + 31) / 32 - 1;
        const CUtensorMap* mX = ti.seg ? &tmXs : (bi == 0 ? &tmX32 : bi == 1 ? &tmX64 : bi == 2 ? &tmX96 : &tmX128);
        const bool gather_x = MODE == 0 && ti.seg == 0;   // the loader warps bring these rows
        const uint32_t x_bytes = gather_x ? 0u : (ti.seg ? (uint32_t)P_X_ROWS : (uint32_t)(bi + 1) * 32u) * 128u;
        const int x_row = ti.row0 + rank * half + ti.group_local * sg.a_group_stride;
        const CUtensorMap* mW0 = ti.seg ? &tmW0_s : &tmW0_r;
        const CUtensorMap* mW1 = ti.seg ? &tmW1_s : &tmW1_r;
        const int w_y = ti.group_local * sg.b_rows_per_group + (MODE == 0 ? ti.nb * 128 + rank * 64 : ti.nb * 256 + rank * 128);
        // weights of a routed expert whose rows fit one tile are read exactly once: let them leave L2 first (1 % of a layer of
        // 3,584 tokens)
        const bool stream_w = ti.seg == 0 && ti.single;
        // the next tile is claimed when 16 k-blocks of this one are left to ask for: a claim takes a few microseconds (an
        // atomic, the M-tile list, the partner's mailbox), and sixteen stages of operands outlast them
        const int kb_pace = max(sg.k_blocks - 16, 0);
        for (int kb = 0; kb < sg.k_blocks; ++kb) {
          if (leader && weights && kb == kb_pace) *prod_pace = (int)it + 1;
          if (!mbar_wait(&free_bar[stage], phase ^ 1, abort_flag, budget)) { ok = false; break; }
          // On routed tiles the partner's producer of the rows brings nothing.  It arrives all the same, so that no stage is taken without it: were
          // it two turns of the ring behind, it would wait for a phase whose parity has come round again, and for good on the last ones.  (As the first
          // thing behind its wait: a prefill of 3,584 tokens 315.2 -> 316.4 us for the arrival, 320.5 behind the loads' code.)
          if (MODE == 0 && WQ && rows && !leader) mbar_arrive(&xfull_bar[stage]);
          // self-test (fmmoe_test_expire_wait): the leader's weights stop here, and the issuer's wait for them runs out
          if (leader && weights && issued == p.test_withhold_stage) { stop = true; break; }
          ++issued;
          unsigned char* sW = smem + stage * L::W_PITCH;
          unsigned char* sX = smem + L::X_OFF + stage * L::X_PITCH;
          const uint32_t bar = full_leader + stage * 8;
          if (leader && rows) mbar_arrive_expect_tx(&full_bar[stage], 2u * ((WQ ? 0u : (uint32_t)P_W_BYTES) + x_bytes));   // both CTAs' boxes
          if (!WQ) {
            if (stream_w) {
              tma_load_2d_pair_hint(sW, mW0, bar, kb * P_BK, w_y, pol_stream);
              if (MODE == 0) tma_load_2d_pair_hint(sW + L::W_RAW / 2, mW1, bar, kb * P_BK, w_y, pol_stream);
            } else {
              tma_load_2d_pair(sW, mW0, bar, kb * P_BK, w_y);
              if (MODE == 0) tma_load_2d_pair(sW + L::W_RAW / 2, mW1, bar, kb * P_BK, w_y);
            }
          } else if (weights) {       // the bytes are this CTA's converters' to read (the maps count columns in bytes)
            mbar_arrive_expect_tx(&wfull_bar[stage], L::W_RAW);
            if (stream_w) {
              tma_load_2d_hint(sW, mW0, &wfull_bar[stage], kb * P_BK, w_y, pol_stream);
              if (MODE == 0) tma_load_2d_hint(sW + L::W_RAW / 2, mW1, &wfull_bar[stage], kb * P_BK, w_y, pol_stream);
            } else {
              tma_load_2d(sW, mW0, &wfull_bar[stage], kb * P_BK, w_y);
              if (MODE == 0) tma_load_2d(sW + L::W_RAW / 2, mW1, &wfull_bar[stage], kb * P_BK, w_y);
            }
          }
          if (rows && !gather_x) tma_load_2d_pair(sX, mX, bar, kb * P_BK, x_row);
          if (++stage == n_stages) { stage = 0; phase ^= 1; }
        }
      }
      // the leader's commits arrive here from another SM: stay until the last of them has
      for (int i = 0; i < n_stages && ok && !stop; ++i) {
        ok = mbar_wait(&free_bar[stage], phase ^ 1, abort_flag, budget);
        if (++stage == n_stages) { stage = 0; phase ^= 1; }
      }
      if (rows) { done[0] = n_kb; done[1] = (int)it; }
      if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
    }
  } else if (warp == 6) {
    // ------------------------------------------------------------ tile scheduler
    // The leader's claims tiles, decodes them and publishes them in its ring and in the partner's mailbox; the partner's moves
    // them from the mailbox into its ring, so that the cluster-scope release and acquire (about a microsecond) are paid here,
    // ahead of time, and no other role waits on anything but its own CTA's ring.
    if (elect_one()) {
      bool ok = true;
      if (leader) {
        const uint32_t mail = cluster_map_shared(smem_u32(const_cast<int*>(mailbox)), 1);
        const uint32_t mfull_partner = cluster_map_shared(smem_u32(mfull_bar), 1);
        uint32_t seq = 0;
        for (; ok; ++seq) {
          if (seq >= 1) {     // the producer says when
            const uint64_t t0 = global_timer_ns();
            while (*prod_pace < (int)seq) {
              __nanosleep(64);
              if (*abort_flag || global_timer_ns() - t0 > budget) { ok = false; break; }
            }
            if (!ok) break;
          }
          // the first tile is the pair's own number: one round trip to memory less in front of the first load
          const int n_pairs = (int)(gridDim.x >> 1);
          const int raw_id = seq == 0 ? (int)(blockIdx.x >> 1) : n_pairs + atomicAdd(p.tile_counter, 1);
          const int tile = raw_id < total_tiles ? raw_id : -1;
          TileInfo ti = {};
          if (tile >= 0) ti = decode_tile(p, MODE, tile, n_mt_r);
          const int slot = seq % G_SCHED;
          const uint32_t sph = ((seq / G_SCHED) & 1) ^ 1;
          if (!mbar_wait(&mempty_bar[slot], sph, abort_flag, budget)) { ok = false; break; }
          const uint32_t m = mail + slot * G_SLOT_INTS * 4;
          st_cluster_u32(m, (uint32_t)tile); st_cluster_u32(m + 4, (uint32_t)ti.seg); st_cluster_u32(m + 8, (uint32_t)ti.group_local);
          st_cluster_u32(m + 12, (uint32_t)ti.row0); st_cluster_u32(m + 16, (uint32_t)ti.rows); st_cluster_u32(m + 20, (uint32_t)ti.nb);
          st_cluster_u32(m + 24, (uint32_t)slot_flags(ti));
          mbar_arrive_cluster(mfull_partner + slot * 8);
          if (!mbar_wait(&sempty_bar[slot], sph, abort_flag, budget)) { ok = false; break; }
          slot_store(ring + slot * G_SLOT_INTS, tile, ti);
          mbar_arrive(&sfull_bar[slot]);
          if (tile < 0) break;
        }
        // the partner's arrivals for the last slots
        for (int i = 0; i < G_SCHED && ok; ++i) { ++seq; ok = mbar_wait(&mempty_bar[seq % G_SCHED], ((seq / G_SCHED) & 1) ^ 1, abort_flag, budget); }
      } else {
        const uint32_t mempty_leader = cluster_map_shared(smem_u32(mempty_bar), 0);
        for (uint32_t seq = 0; ok; ++seq) {
          const int slot = seq % G_SCHED;
          const uint32_t sph = (seq / G_SCHED) & 1;
          if (!mbar_wait_cluster(&mfull_bar[slot], sph, abort_flag, budget)) { ok = false; break; }
          const int tile = mailbox[slot * G_SLOT_INTS];
          const TileInfo ti = slot_load(mailbox + slot * G_SLOT_INTS);
          if (!mbar_wait(&sempty_bar[slot], sph ^ 1, abort_flag, budget)) { ok = false; break; }
          slot_store(ring + slot * G_SLOT_INTS, tile, ti);
          mbar_arrive(&sfull_bar[slot]);
          mbar_arrive_remote(mempty_leader + slot * 8);
          if (tile < 0) break;
        }
      }
      // a scheduler that gave up because another role aborted records nothing: the status word has the cause
      if (!ok && !*abort_flag) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
    }
  } else if (warp == 1) {
    if (leader && elect_one()) {
      // ---------------------------------------------------------- MMA issuer (leader CTA only)
      int stage = 0; uint32_t phase = 0;
      int as = 0; uint32_t aphase = 0;
      int cs = 0; uint32_t cphase = 0;
      bool ok = true;
      for (uint32_t it = 0; ok; ++it) {
        TileInfo ti;
        if (!wait_tile(it, ti, ok)) break;
        release_tile(it);
        const uint32_t idesc = umma_idesc_bf16(256, pair_n_pad(ti.rows));
        const int k_blocks = p.seg[MODE][ti.seg].k_blocks;
        if (!mbar_wait(&tempty_bar[as], aphase ^ 1, abort_flag, budget)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + as * 256;
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (!mbar_wait(&full_bar[stage], phase, abort_flag, budget)) { ok = false; break; }
          if (WQ && !mbar_wait(&cfull_bar[cs], cphase, abort_flag, budget)) { ok = false; break; }
          if (MODE == 0) fence_proxy_async_smem();   // rows written by the loader warps' cp.async
          tc_fence_after();
          const uint64_t dw = umma_desc_sw128(smem_u32(WQ ? smem + L::CVT_OFF + cs * P_W_BYTES : smem + stage * L::W_PITCH));
          const uint64_t dx = umma_desc_sw128(smem_u32(smem + L::X_OFF + stage * L::X_PITCH));
#pragma unroll
          for (int k = 0; k < P_BK / 16; ++k)
            umma_bf16_pair(d_tmem, dw + 2 * k, dx + 2 * k, idesc, (kb | k) != 0);
          umma_commit_pair_multicast(&empty_bar[stage], 3);   // both CTAs' stage is reusable once these MMAs have read it
          if (++stage == L::X_STAGES) { stage = 0; phase ^= 1; }
          if (WQ) {
            umma_commit_pair_multicast(&cempty_bar[cs], 3);   // and so are the expanded weights
            if (++cs == L::CVT_STAGES) { cs = 0; cphase ^= 1; }
          }
        }
        if (!ok) break;
        umma_commit_pair_multicast(&tfull_bar[as], 3);        // accumulator complete, in both CTAs
        if (++as == 2) { as = 0; aphase ^= 1; }
      }
      // the partner's arrivals for the last accumulators
      for (int i = 0; i < 2 && ok; ++i) {
        ok = mbar_wait(&tempty_bar[as], aphase ^ 1, abort_flag, budget);
        if (++as == 2) { as = 0; aphase ^= 1; }
      }
      if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
    } else if (MODE == 0 && !leader && elect_one()) {
      // ---------------------------------------------------------- relay (partner, GEMM-1): cp.async can only signal its own CTA
      const uint32_t full_leader = cluster_map_shared(smem_u32(full_bar), 0);
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      for (uint32_t it = 0; ok; ++it) {
        TileInfo ti;
        if (!wait_tile(it, ti, ok)) break;
        release_tile(it);
        const int k_blocks = p.seg[MODE][ti.seg].k_blocks;
        for (int kb = 0; kb < k_blocks; ++kb) {
          if (!mbar_wait(&xfull_bar[stage], phase, abort_flag, budget)) { ok = false; break; }
          fence_proxy_async_smem();
          mbar_arrive_remote(full_leader + stage * 8);
          if (++stage == L::X_STAGES) { stage = 0; phase ^= 1; }
        }
      }
      if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
    }
  } else if (MODE == 0 && warp >= P_BASE_THREADS / 32 && warp < (P_BASE_THREADS + P_LOADERS) / 32) {
    // ------------------------------------------------------------ row loaders (GEMM-1, warps 7-10, both CTAs)
    // Every stage of a routed tile: this CTA's half of its rows x 128 bytes of x, row r = token row_token[row0 + rank * half + r],
    // written where a TMA box with the 128-byte swizzle would put them (16-byte chunk c of row r at r*128 + ((c ^ (r & 7)) * 16)).
    // Eight lanes cover one row, a thread serves rows q, q+16, ...  For other tiles they only keep the stage barriers in step.
    const int lt = threadIdx.x - P_BASE_THREADS;            // 0..127
    const int chunk = lt & 7, rq = lt >> 3;            // rq 0..15
    const uint32_t dst0 = (uint32_t)(L::X_OFF + rq * 128 + ((chunk ^ (rq & 7)) << 4));
    uint64_t* landed = leader ? full_bar : xfull_bar;
    int stage = 0; uint32_t phase = 0;
    bool ok = true;
    const __nv_bfloat16* xg = p.x + chunk * 8;
    for (uint32_t it = 0; ok; ++it) {
      TileInfo ti;
      if (!wait_tile(it, ti, ok, true)) break;
      __syncwarp();
      if (lane == 0) release_tile(it);
      const bool gather_x = ti.seg == 0;
      const int half = pair_n_pad(ti.rows) >> 1, first = rank * half;
      const __nv_bfloat16* src[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = rq + 16 * i;
        src[i] = gather_x && r < half && first + r < ti.rows ? xg + (long long)p.row_token[ti.row0 + first + r] * p.ld_x : nullptr;
      }
      const int k_blocks = p.seg[MODE][ti.seg].k_blocks;
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait_warp(&empty_bar[stage], phase ^ 1, abort_flag, budget)) { ok = false; break; }
        if (gather_x) {
          const uint32_t sX = smem_u32(smem + stage * L::X_PITCH) + dst0;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (src[i]) cp_async_16(sX + i * 2048, src[i] + kb * P_BK);
          cp_async_arrive_noinc(&landed[stage]);
        } else {
          mbar_arrive(&landed[stage]);
        }
        if (++stage == L::X_STAGES) { stage = 0; phase ^= 1; }
      }
    }
    if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
  } else if (WQ && warp >= (pair_threads<MODE, WQ>() - P_CONVERTERS) / 32 - 1) {
    // ------------------------------------------------------------ weight converters (FP8 stream, the last eight warps but one, both CTAs)
    // Per k-block: 128 rows x 64 FP8 bytes (64-byte rows) -> 128 rows x 64 bf16 in the 128-byte swizzle.  A thread takes 16 bytes
    // (row p/4, bytes 16*(p%4) ..) at a time: one 16-byte load, two 16-byte stores; consecutive threads read consecutive pieces
    // and the eight lanes of a quarter-warp write eight different chunks.  Two groups take alternate k-blocks, so that one group's
    // waits, loads and proxy fence pass under the other's arithmetic.
    const int ct = (int)threadIdx.x - (pair_threads<MODE, WQ>() - P_CONVERTERS - 32), grp = ct >> 7, gt = ct & 127;
    const uint32_t cfull_leader = cluster_map_shared(smem_u32(cfull_bar), 0);
    int stage = grp; uint32_t phase = 0;
    int cs = grp; uint32_t cphase = 0;
    bool ok = true;
    for (uint32_t it = 0; ok; ++it) {
      TileInfo ti;
      if (!wait_tile(it, ti, ok, true)) break;
      __syncwarp();
      if (lane == 0) release_tile(it);
      const Segment& sg = p.seg[MODE][ti.seg];
      // block scales: rows 0-63 and 64-127 of this CTA's 128 (GEMM-1: gate and up rows of one feature block); lane l holds the
      // exponent of 128-column block l of 32
      const int n_kb128 = (sg.k_blocks + 1) >> 1, rb_per_group = (sg.b_rows_per_group + 127) >> 7;
      const int rb = MODE == 0 ? ti.nb : 2 * ti.nb + rank;
      const long long sc_row = ((long long)ti.group_local * rb_per_group + min(rb, rb_per_group - 1)) * n_kb128;
      int se0 = 0, se1 = 0;
      for (int kb = grp; kb < sg.k_blocks; kb += 2) {      // k_blocks is even: FP8 layers come in whole 128-column blocks
        if (((kb >> 1) & 31) == 0 && (kb >> 1) + lane < n_kb128) {
          se0 = p.wscale[MODE][ti.seg][0][sc_row + (kb >> 1) + lane];
          se1 = MODE == 0 ? p.wscale[MODE][ti.seg][1][sc_row + (kb >> 1) + lane] : se0;
        }
        // warp-uniform outcome: the arrivals below are made by one lane on behalf of the warp
        if (!__all_sync(0xffffffffu, mbar_wait(&wfull_bar[stage], phase, abort_flag, budget) &&
                                     mbar_wait(&cempty_bar[cs], cphase ^ 1, abort_flag, budget))) { ok = false; break; }
        const int e0 = __shfl_sync(0xffffffffu, se0, (kb >> 1) & 31), e1 = __shfl_sync(0xffffffffu, se1, (kb >> 1) & 31);
        const unsigned char* raw_w = smem + stage * L::W_PITCH + gt * 16;
        // piece i * 128 + gt: row i * 32 + gt / 4, whose swizzle does not depend on i
        const int r0 = gt >> 2, c0 = gt & 3;
        unsigned char* out_w = smem + L::CVT_OFF + cs * P_W_BYTES + r0 * 128;
        uint4 q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = *reinterpret_cast<const uint4*>(raw_w + i * 2048);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t mbits = (uint32_t)(247 + (i < 2 ? e0 : e1)) << 7;      // bf16 2^(120 + scale exponent)
          const uint32_t m2 = mbits | (mbits << 16);
          const __nv_bfloat162 mul = *reinterpret_cast<const __nv_bfloat162*>(&m2);
          uint4 o0, o1;
          e4m3x4_to_bf16x4(q[i].x, mul, o0.x, o0.y); e4m3x4_to_bf16x4(q[i].y, mul, o0.z, o0.w);
          e4m3x4_to_bf16x4(q[i].z, mul, o1.x, o1.y); e4m3x4_to_bf16x4(q[i].w, mul, o1.z, o1.w);
          *reinterpret_cast<uint4*>(out_w + i * 4096 + (((2 * c0) ^ (r0 & 7)) << 4)) = o0;
          *reinterpret_cast<uint4*>(out_w + i * 4096 + (((2 * c0 + 1) ^ (r0 & 7)) << 4)) = o1;
        }
        fence_proxy_async_smem();            // the MMA reads these generic-proxy writes through the async proxy
        __syncwarp();
        if (lane == 0) {
          if (leader) mbar_arrive(&cfull_bar[cs]);
          else mbar_arrive_remote(cfull_leader + cs * 8);
          mbar_arrive(&wempty_bar[stage]);   // this warp is done with the stage's weight bytes
        }
        if ((stage += 2) >= L::W_STAGES) { stage -= L::W_STAGES; phase ^= 1; }
        if ((cs += 2) >= L::CVT_STAGES) { cs -= L::CVT_STAGES; cphase ^= 1; }
      }
    }
    // The leader's commits for the last three buffers.  The next k-block's buffer would be free behind the third last k-block's
    // commit, the one after it behind the second last's, the third behind the last's: the first and the third are group 0's.
    for (int i = 0; i < (grp ? 1 : 2) && ok; ++i) {
      ok = mbar_wait_warp(&cempty_bar[cs], cphase ^ 1, abort_flag, budget);
      if ((cs += 2) >= L::CVT_STAGES) { cs -= L::CVT_STAGES; cphase ^= 1; }
    }
    if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
  } else {
    // ------------------------------------------------------------ epilogue (both CTAs, own 128 weight rows)
    // Two sets of four warps (2-5 and the four behind the loaders) take alternate 32-token blocks of a tile.
    const int set = warp >= 6;
    const int q = warp & 3;                 // TMEM lane quarter this warp may access = weight rows 32q .. 32q+31 of this CTA
    const uint32_t tempty_leader = cluster_map_shared(smem_u32(tempty_bar), 0);
    int as = 0; uint32_t aphase = 0;
    uint32_t xc = 0;                        // GEMM-1: 32-token blocks swapped so far
    bool ok = true;
    for (uint32_t it = 0; ok; ++it) {
      TileInfo ti;
      if (!wait_tile(it, ti, ok, true)) break;
      __syncwarp();
      if (lane == 0) release_tile(it);
      const Segment& sg = p.seg[MODE][ti.seg];
      float gate[4];                        // GEMM-2: gates of this set's rows, lane l: row 32 c + l of block c; asked for early
      if (MODE == 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = (2 * i + set) * 32 + lane;
          gate[i] = ti.seg == 0 && !p.deterministic && r < ti.rows ? p.row_gate[ti.row0 + r] : 1.f;
        }
      }
      if (!mbar_wait_warp(&tfull_bar[as], aphase, abort_flag, budget)) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + as * 256 + (static_cast<uint32_t>(q * 32) << 16);
      const long long out_row0 = (long long)ti.row0 + (long long)ti.group_local * sg.out_group_stride;
      const int n_chunks = (ti.rows + 31) >> 5;
      if (MODE == 0) {
        const bool up = q >= 2;             // this warp holds up rows; its feature block's gate rows are warp q - 2's
        const int feat0 = ti.nb * 128 + rank * 64 + (q & 1) * 32;
        const bool f_ok = feat0 < sg.n_valid;      // a multiple of 64: all 32 features or none
        __nv_bfloat16* dst = p.act[ti.seg] + (out_row0 + (up ? 16 : 0)) * sg.ld_out + feat0;
        const int sw = (lane >> 1) & 3;     // 16-byte pieces of a lane's 64 bytes, permuted so that eight lanes meet eight bank groups
#pragma unroll 1
        for (int c = set; c < n_chunks; c += 2, ++xc) {
          uint32_t v[32];
          tmem_ld32(taddr + c * 32, v);
          tmem_ld_wait();
          const int b = (int)(xc & 1);
          float4* mine = reinterpret_cast<float4*>(xch + ((set * 4 + q) * 2 + b) * 512) + lane * 4;
          const float4* theirs = reinterpret_cast<const float4*>(xch + ((set * 4 + (q ^ 2)) * 2 + b) * 512) + lane * 4;
          uint64_t* swapped = &xch_bar[(set * 2 + (q & 1)) * 2 + b];
          // the half of the block the other warp finishes: a gate warp finishes tokens 0-15, an up warp 16-31
          float keep[16];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float4 g;
            g.x = __uint_as_float(up ? v[4 * i] : v[16 + 4 * i]); g.y = __uint_as_float(up ? v[4 * i + 1] : v[17 + 4 * i]);
            g.z = __uint_as_float(up ? v[4 * i + 2] : v[18 + 4 * i]); g.w = __uint_as_float(up ? v[4 * i + 3] : v[19 + 4 * i]);
            mine[i ^ sw] = g;
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) keep[i] = __uint_as_float(up ? v[16 + i] : v[i]);
          __syncwarp();
          if (lane == 0) mbar_arrive(swapped);
          if (!mbar_wait_warp(swapped, (xc >> 1) & 1, abort_flag, budget)) { ok = false; break; }
          float a[16];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 o4 = theirs[i ^ sw];
            const float o[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float g0 = up ? o[j] : keep[4 * i + j], u0 = up ? keep[4 * i + j] : o[j];
              a[4 * i + j] = __fdividef(g0, 1.f + __expf(-g0)) * u0;
            }
          }
          const int nt = f_ok ? ti.rows - c * 32 - (up ? 16 : 0) : 0;      // rows to store among this warp's sixteen
          store_rows_bf16<16>(dst + (long long)(c * 32) * sg.ld_out, sg.ld_out, a, nt, lane);
        }
        if (!ok) break;
      } else {
        const int feat0 = ti.nb * 256 + rank * 128 + q * 32;
        const bool f_ok = feat0 < sg.n_valid;
        float* gates = xch + (set * 4 + q) * 32;
#pragma unroll 1
        for (int c = set; c < n_chunks; c += 2) {
          const int nt = f_ok ? min(32, ti.rows - c * 32) : 0;      // rows to write, warp-uniform
          const float gate_c = c < 2 ? gate[0] : c < 4 ? gate[1] : c < 6 ? gate[2] : gate[3];   // 1 in fixed-order mode: gates are applied by the ordered gather
          uint32_t v[32];
          tmem_ld32(taddr + c * 32, v);
          if (p.pair) {
            // pair-row mode: gate-scaled bf16 rows per pair
            gates[lane] = gate_c;
            __syncwarp();
            tmem_ld_wait();
            float a[32];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float4 g4 = reinterpret_cast<const float4*>(gates)[i];
              a[4 * i] = g4.x * __uint_as_float(v[4 * i]); a[4 * i + 1] = g4.y * __uint_as_float(v[4 * i + 1]);
              a[4 * i + 2] = g4.z * __uint_as_float(v[4 * i + 2]); a[4 * i + 3] = g4.w * __uint_as_float(v[4 * i + 3]);
            }
            store_rows_bf16<32>(p.yb[ti.seg] + (out_row0 + c * 32) * sg.ld_out + feat0, sg.ld_out, a, nt, lane);
            __syncwarp();
          } else if (p.deterministic) {
            tmem_ld_wait();
            float* yb = p.y[ti.seg] + (out_row0 + c * 32) * sg.ld_out + feat0 + lane;
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (j < nt) yb[(long long)j * sg.ld_out] = __uint_as_float(v[j]);
          } else {
            tmem_ld_wait();
            const int tok_l = ti.seg ? ti.row0 + c * 32 + lane : lane < nt ? p.row_token[ti.row0 + c * 32 + lane] : 0;
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const int tk = __shfl_sync(0xffffffffu, tok_l, j);
              const float gt = __shfl_sync(0xffffffffu, gate_c, j);
              if (j < nt) atomicAdd(p.acc + (long long)tk * sg.ld_out + feat0 + lane, gt * __uint_as_float(v[j]));
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (leader) mbar_arrive(&tempty_bar[as]);
        else mbar_arrive_remote(tempty_leader + as * 8);
      }
      if (++as == 2) { as = 0; aphase ^= 1; }
    }
    if (!ok) { atomicCAS(p.status, 0, DEV_TIMEOUT); *abort_flag = 1; }
  }

  // ---------------------------------------------------------------- teardown
  // The next kernel of the stream may be scheduled from here on, not earlier: its CTAs then meet SMs that this
  // grid is about to leave, instead of sitting beside a pair whose tensor memory is still bound to two SMs.
  pdl_launch_dependents();
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  const bool gave_up = *abort_flag != 0;
  auto let_land = [&]() {      // give copies and arrivals still in flight time to land before the shared memory is released
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 200000ull) { }
    __syncthreads();
  };
  if (gave_up) {
    let_land();
  } else if (p.check_drained && threadIdx.x == 0) {
    // self-check: barrier i of a ring of n has completed as many phases as uses it has seen
    auto drained = [&](uint64_t* bar, int n, int uses) {
      bool all = true;
      for (int i = 0; i < n; ++i) all &= mbar_test_wait(&bar[i], (uint32_t)((uses > i ? (uses - i + n - 1) / n : 0) - 1) & 1u);
      return all;
    };
    bool all = drained(empty_bar, L::X_STAGES, done[0]);
    if (WQ) all &= drained(cempty_bar, L::CVT_STAGES, done[0]);
    if (leader) all &= drained(tempty_bar, 2, done[1]) && drained(mempty_bar, G_SCHED, done[1] + 1);
    if (!all) atomicCAS(p.status, 0, DEV_INTERNAL);
  }
  // Neither CTA may release its shared or tensor memory while the other's loads, commits and arrivals can still touch it.
  // Everything that a CTA is sent is awaited by a role of that CTA before it comes here: the loads' bytes and the partner's rows and
  // weights by the issuer with their stage, the commits on a stage by its producer, on expanded weights by the converters, on an
  // accumulator by the epilogue, the partner's arrivals on accumulators by the issuer, the mailbox's by the schedulers.  So
  // the barrier, at which both CTAs meet before the pair's tensor memory goes, need not order any of it (an arrival with release
  // would first wait for the epilogue's last stores).  A CTA that gave up has not awaited it all: it lets it land once more
  // behind the barrier, before which the other sent its last.
  cluster_arrive_relaxed();
  cluster_wait();
  if (gave_up) let_land();
  if (warp == 1) {
    tc_fence_after();
    tmem_relinquish_pair();
    tmem_dealloc_pair(tmem_base, P_TMEM_COLS);
  }
}

// ---------------------------------------------------------------- host side
template <int WQ>
static fmmoe_status launch_ffn_tc2_impl(fmmoe_handle* h, const FfnArgs& a, cudaStream_t s) {
  using L = PairLayout<WQ>;
  const fmmoe_layer_desc& d = *a.d;
  const int H = d.hidden, I = d.inter, E = d.n_experts, Ns = d.n_shared, Is = d.shared_inter;
  if (!h->encode_tiled) return FMMOE_ERR_CUDA;
  if (a.T == 0) return FMMOE_OK;
  const int mtps = (int)((a.T + PAIR_BLOCK_M - 1) / PAIR_BLOCK_M);
  const uint64_t p_rows = (uint64_t)a.p_max;

  CUtensorMap X2r[4], X1s, X2s, G1r, U1r, G1s, U1s, D2r, D2s;
  bool ok = true;
  auto wmap = [&](CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
    return WQ ? make_map_u8(h, m, base, rows, cols, box_rows) : make_map(h, m, base, rows, cols, box_rows);
  };
  for (int i = 0; i < 4; ++i) ok &= make_map(h, &X2r[i], a.act, p_rows, I, 32 * (i + 1));
  ok &= wmap(&G1r, a.w->w_gate, (uint64_t)E * I, H, 64);
  ok &= wmap(&U1r, a.w->w_up, (uint64_t)E * I, H, 64);
  ok &= wmap(&D2r, a.w->w_down, (uint64_t)E * H, I, 128);
  if (Ns) {
    ok &= make_map(h, &X1s, a.x, (uint64_t)a.T, H, P_X_ROWS);
    ok &= wmap(&G1s, a.w->ws_gate, (uint64_t)Ns * Is, H, 64);
    ok &= wmap(&U1s, a.w->ws_up, (uint64_t)Ns * Is, H, 64);
    ok &= make_map(h, &X2s, a.act_sh, (uint64_t)Ns * a.T, Is, P_X_ROWS);
    ok &= wmap(&D2s, a.w->ws_down, (uint64_t)Ns * H, Is, 128);
  } else {
    X1s = X2r[0]; G1s = G1r; U1s = U1r; X2s = X2r[0]; D2s = D2r;   // never dereferenced without shared experts
  }
  if (!ok) return FMMOE_ERR_CUDA;

  GemmParams p = {};
  p.mtiles = a.mtiles; p.n_mtiles = a.n_mtiles; p.max_mtiles = a.max_mtiles;
  p.block_m = PAIR_BLOCK_M; p.shared_mtiles = Ns * mtps; p.mt_per_shared = mtps; p.rows_major = 1; p.T = a.T;
  p.seg[0][0] = Segment{(I + 127) / 128, H / P_BK, I, I, 0, 0, I};
  p.seg[0][1] = Segment{Ns ? (Is + 127) / 128 : 0, H / P_BK, Is, Is, 0, (int)a.T, Is};
  p.seg[1][0] = Segment{(H + 255) / 256, I / P_BK, H, H, 0, 0, H};
  p.seg[1][1] = Segment{Ns ? (H + 255) / 256 : 0, Ns ? Is / P_BK : 0, H, H, (int)a.T, (int)a.T, H};
  fill_params(p, a);
  p.wait_budget_ns = h->wait_budget_ns; p.check_drained = h->debug_sync;
  p.tile_counter = a.tile_counters; p.test_withhold_stage = a.test_withhold_stage;
  GemmParams p2 = p;
  p2.tile_counter = a.tile_counters + 1; p2.test_withhold_stage = -1;

  bool& attr_set = WQ ? h->tc2q_attr_set : h->tc2_attr_set;
  if (!attr_set) {
    FMMOE_CUDA_TRY(cudaFuncSetAttribute(ffn_tc2_kernel<0, WQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM_BYTES));
    FMMOE_CUDA_TRY(cudaFuncSetAttribute(ffn_tc2_kernel<1, WQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM_BYTES));
    attr_set = true;
  }
  const int grid = a.grid_override > 0 ? 2 * a.grid_override : h->sm_count & ~1;      // whole CTA pairs
  { ProfScope ps(h, FMMOE_KERNEL_GEMM1, s); FMMOE_CUDA_TRY(launch_ex(ffn_tc2_kernel<0, WQ>, dim3(grid), dim3((pair_threads<0, WQ>())), L::SMEM_BYTES, s, 2, false, X2r[0], X2r[1], X2r[2], X2r[3], X1s, G1r, U1r, G1s, U1s, p)); }
  FMMOE_CUDA_TRY(cudaGetLastError());
  { ProfScope ps(h, FMMOE_KERNEL_GEMM2, s); FMMOE_CUDA_TRY(launch_ex(ffn_tc2_kernel<1, WQ>, dim3(grid), dim3((pair_threads<1, WQ>())), L::SMEM_BYTES, s, 2, false, X2r[0], X2r[1], X2r[2], X2r[3], X2s, D2r, D2r, D2s, D2s, p2)); }
  FMMOE_CUDA_TRY(cudaGetLastError());
  h->launches += 2;
  return FMMOE_OK;
}

fmmoe_status launch_ffn_tc2(fmmoe_handle* h, const FfnArgs& a, cudaStream_t s) {
  return a.d->weight_format == FMMOE_WEIGHTS_FP8_BLOCK128 ? launch_ffn_tc2_impl<1>(h, a, s) : launch_ffn_tc2_impl<0>(h, a, s);
}

}  // namespace fmmoe
