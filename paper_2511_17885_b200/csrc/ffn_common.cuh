// Pieces shared by the two forms of the grouped expert GEMM, both with the token rows as the MMA's N dimension (ffn_sm.cu: one
// CTA a tile, up to 128 rows; ffn_tc2.cu: CTA pairs, up to 256 rows): the tile list arithmetic, the decoded-tile ring slot, the
// store of an epilogue's rows, the FP8 expansion and the tensor-map helper.
#pragma once
#include <cuda_bf16.h>

#include "internal.h"
#include "ptx.cuh"

namespace fmmoe {

constexpr int G_SCHED = 4;         // slots of the tile ring
constexpr int G_SLOT_INTS = 8;     // a slot: tile id (-1: no more tiles) + the decoded TileInfo

struct Segment {          // routed experts (0) or shared experts (1)
  int n_nblocks;          // N-blocks per group
  int k_blocks;           // K / 64
  int b_rows_per_group;   // rows of the B tensor per group (S_m for GEMM-1, H for GEMM-2)
  int n_valid;            // valid output columns per group (S_m for GEMM-1, H for GEMM-2)
  int a_group_stride;     // rows added to the A row per group index (shared experts only)
  int out_group_stride;   // rows added to the output row per group index
  int ld_out;             // leading dimension of the output (elements)
};

// Phase 0: GEMM-1 + SwiGLU, phase 1: GEMM-2 + combine.  The small-M form does both in one launch, CTA pairs launch them one by one.
struct GemmParams {
  const MTile* mtiles;        // routed M-tiles
  const int32_t* n_mtiles;    // device: number of routed M-tiles
  int max_mtiles;             // capacity of `mtiles` (a corrupt count must not walk past it)
  int32_t* tile_counter;      // device: next tile to hand out (zero at launch)
  int phases;                 // small-M form: bit 0: GEMM-1's tiles, bit 1: GEMM-2's (one launch each when kernels are timed one by one)
  int32_t* gave_up;           // device, small-M form: set when a CTA of this call gives up (zero at launch)
  int32_t* done;              // device, small-M form: arrivals per M-tile, routed ones, then (from max_mtiles on) shared ones; zero at launch
  int block_m;                // rows per M-tile of the tile list (128; 256 for CTA pairs)
  int shared_mtiles;          // N_s * ceil(T/block_m), host-known
  int mt_per_shared;          // ceil(T/block_m)
  long long T;
  Segment seg[2][2];          // [phase][segment]
  // epilogue
  __nv_bfloat16* act[2];      // GEMM-1: activation outputs (routed, shared)
  const __nv_bfloat16* x; int ld_x;   // GEMM-1: hidden states [T, H] the routed rows are gathered from
  const int32_t* row_token;   // grouped row -> token (GEMM-1: gather, GEMM-2: combine)
  const float* row_gate;      // GEMM-2
  float* acc;                 // GEMM-2 atomic:  [T, H]
  float* y[2];                // GEMM-2 deterministic: routed [P, H], shared [N_s*T, H]
  __nv_bfloat16* yb[2];       // GEMM-2 pair-row mode: gate-scaled outputs per pair, bf16, same shapes
  int deterministic;
  int pair;                   // GEMM-2: write yb instead of reducing into acc
  int* status;
  const int8_t* wscale[2][2][2];       // FP8 weight stream: block scale exponents, [phase][segment][weight box of the stage]
  unsigned long long wait_budget_ns;   // time budget of every bounded wait
  int rows_major;                      // shared-expert tiles M-tile-major too
  int shared_first;                    // GEMM-1, small-M form: so many shared-expert tiles come before all others
  int routed_first;                    // GEMM-2, small-M form: so many routed tiles come before the others: the shared experts' activations are GEMM-1's last
  int fine;                            // GEMM-2, small-M form: tiles of 128 features, two k-blocks a stage
  int test_withhold_stage;             // self-test: the producer stops before this k-block (-1: never)
  int check_drained;                   // CTA pairs, self-check: nothing that was sent to a CTA is still under way when it leaves
};

// Four E4M3 bytes -> four bf16 in two words, times `mul` (a power of two in both halves).  An E4M3 byte s.eeee.mmm placed as
// s.0000eeee.mmm0000 is the bf16 number 2^(e-127) (1 + m/8), or the bf16 subnormal 2^-126 (m/8) for e = 0: in both cases the
// E4M3 value times 2^-120, so one exact bf16 multiply by 2^(120 + scale exponent) finishes the conversion.  The upper bytes
// (s0000eee) and the lower bytes (emmm0000) of all four are made at once and then interleaved.
__device__ __forceinline__ void e4m3x4_to_bf16x4(uint32_t w, __nv_bfloat162 mul, uint32_t& o0, uint32_t& o1) {
  const uint32_t hi = ((w >> 4) & 0x07070707u) | (w & 0x80808080u);
  const uint32_t lo = (w << 4) & 0xf0f0f0f0u;
  const uint32_t a = __byte_perm(hi, lo, 0x1504), b = __byte_perm(hi, lo, 0x3726);
  const __nv_bfloat162 va = __hmul2(*reinterpret_cast<const __nv_bfloat162*>(&a), mul);
  const __nv_bfloat162 vb = __hmul2(*reinterpret_cast<const __nv_bfloat162*>(&b), mul);
  o0 = *reinterpret_cast<const uint32_t*>(&va);
  o1 = *reinterpret_cast<const uint32_t*>(&vb);
}

struct TileInfo {
  int phase, seg, group_local, row0, rows, nb;
  int dep;       // entry of `done`: GEMM-1 adds to it, GEMM-2 waits for it
  bool single;   // routed: the expert's rows fit this one M-tile
  bool ready;    // GEMM-2: the activations were there when the tile was handed out
};

// Number of routed M-tiles, and one of them.  Read from L2: a line of an older call may still be in L1.
__device__ __forceinline__ int routed_mtiles(const GemmParams& p) { return p.n_mtiles ? min(max(__ldcg(p.n_mtiles), 0), p.max_mtiles) : 0; }
__device__ __forceinline__ MTile load_mtile(const MTile* m) {
  const int4 v = __ldcg(reinterpret_cast<const int4*>(m));
  return MTile{v.x, v.y, v.z, v.w};
}
// Tiles of a phase.
__device__ __forceinline__ int phase_tiles(const GemmParams& p, int phase, int n_mt_r) {
  return n_mt_r * p.seg[phase][0].n_nblocks + p.shared_mtiles * p.seg[phase][1].n_nblocks;
}

// Tile `tile` of a phase -> (segment, M-tile, N-block).  Routed tiles M-tile-major, the shared experts' interleaved with them evenly
// behind the ones that come first.  Those go N-block-major in the small-M form, so that the CTAs running at the same time share a weight
// tile, and M-tile-major with CTA pairs, where the rows are what does not fit L2, not the few shared weights.  19,456 tokens of
// the 64-expert layer, N-block-major / M-tile-major: DRAM reads of GEMM-1 2.44 / 1.16 GB, of GEMM-2 1.43 / 0.67 GB, the layer 1,690 / 1,536 us in a
// sustained loop (under the power cap bytes are time); 4,864 tokens 496 / 495, 2,432 no difference.
__device__ __forceinline__ TileInfo decode_tile(const GemmParams& p, int phase, int tile, int n_mt_r) {
  TileInfo ti;
  ti.phase = phase;
  ti.ready = false;
  const Segment* sg = p.seg[phase];
  int r = tile;            // routed tile, or
  int t2 = -1;             // shared tile
  if (p.shared_mtiles) {   // else no interleaving, no 64-bit divisions
    const int R = n_mt_r * sg[0].n_nblocks, S = p.shared_mtiles * sg[1].n_nblocks;
    const int lead_s = phase ? 0 : p.shared_first, lead_r = phase ? min(R, p.routed_first) : 0;
    const int pos = tile - lead_s - lead_r;
    if (pos < 0) {
      if (!phase) t2 = tile;
    } else {
      const unsigned long long s = (unsigned long long)(S - lead_s), n = s + (unsigned long long)(R - lead_r);
      const int sb = (int)((unsigned long long)pos * s / n);           // shared tiles before this position
      const int sb1 = (int)((unsigned long long)(pos + 1) * s / n);
      if (sb1 != sb) t2 = lead_s + sb;
      else r = lead_r + pos - sb;
    }
  }
  if (t2 < 0) {
    const int mt = r / sg[0].n_nblocks;
    ti.seg = 0;
    ti.nb = r - mt * sg[0].n_nblocks;
    const MTile m = load_mtile(p.mtiles + mt);
    ti.group_local = m.group; ti.row0 = m.row0; ti.rows = m.rows;
    ti.single = m.pad != 0;
    ti.dep = mt;
  } else {
    ti.seg = 1;
    const int by = p.rows_major ? sg[1].n_nblocks : p.shared_mtiles, q = t2 / by, rest = t2 - q * by, mt = p.rows_major ? q : rest;
    ti.nb = p.rows_major ? rest : q;
    ti.group_local = mt / p.mt_per_shared;
    const int mb = mt - ti.group_local * p.mt_per_shared;
    ti.row0 = mb * p.block_m;
    const long long left = p.T - (long long)ti.row0;
    ti.rows = left < p.block_m ? (int)left : p.block_m;
    ti.single = false;
    ti.dep = p.max_mtiles + mt;
  }
  return ti;
}

// A slot of the tile ring as the scheduler publishes it and the other roles read it.
__device__ __forceinline__ int slot_flags(const TileInfo& ti) { return (ti.single ? 1 : 0) | (ti.phase << 1) | (ti.ready ? 4 : 0); }
__device__ __forceinline__ void slot_store(volatile int* s, int tile, const TileInfo& ti) {
  s[0] = tile; s[1] = ti.seg; s[2] = ti.group_local; s[3] = ti.row0; s[4] = ti.rows; s[5] = ti.nb; s[6] = slot_flags(ti); s[7] = ti.dep;
}
__device__ __forceinline__ TileInfo slot_load(const volatile int* s) {
  TileInfo ti;
  const int f = s[6];
  ti.seg = s[1]; ti.group_local = s[2]; ti.row0 = s[3]; ti.rows = s[4]; ti.nb = s[5]; ti.dep = s[7];
  ti.single = f & 1; ti.phase = (f >> 1) & 1; ti.ready = (f & 4) != 0;
  return ti;
}

constexpr int DONE_PER_TILE = 4;     // the epilogue warps of a CTA
// What GEMM-1 wrote of an M-tile, for GEMM-2's tensor loads on other SMs.  Writers (a warp that has stored its part of a tile): every
// lane orders its stores before asynchronous reads, one lane publishes them for the warp.  Readers: a thread that has seen the count
// full, and before its first load orders what follows behind it (fence_proxy_async_global).
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }
__device__ __forceinline__ void publish_rows(const GemmParams& p, const TileInfo& ti, int lane) {
  fence_proxy_async_global();
  __syncwarp();
  if (lane == 0) {
    __threadfence();
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p.done + ti.dep) : "memory");
  }
}
__device__ __forceinline__ bool rows_ready(const GemmParams& p, const TileInfo& ti) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p.done + ti.dep) : "memory");
  return v >= p.seg[0][ti.seg].n_nblocks * DONE_PER_TILE;
}
// Bounded; gives up too when another role of this CTA or another CTA of this call has.  (Not by the status word: that may still hold
// what an earlier call or another kernel recorded.)
__device__ __forceinline__ bool wait_rows(const GemmParams& p, const TileInfo& ti, const volatile int* abort_flag, uint64_t budget) {
  const uint64_t t0 = global_timer_ns();
  for (uint32_t spins = 1; !rows_ready(p, ti); ++spins) {
    if (*abort_flag || global_timer_ns() - t0 > budget) return false;
    if ((spins & 63) == 0 && *(const volatile int32_t*)p.gave_up != 0) return false;
    __nanosleep(32);
  }
  return true;
}

// N consecutive token rows of one feature a lane (lanes: 32 consecutive features) -> bf16 rows.  Two exchanges between
// neighbouring lanes leave every lane with four features of one token of four, so that a store instruction writes whole
// 64-byte segments of four rows with 8 bytes a lane.  All exchanges come before the stores: a store under a lane's own
// condition between them made every step wait for the last.  32 rows 1,290 -> 640 clocks; GEMM-2 on 14,336 tokens of the
// 128-expert layer, which waited for its epilogue 23 % of the time, 221.8 k -> 196.7 k clocks.  Rows from nt on are not written.
template <int N>
__device__ __forceinline__ void store_rows_bf16(__nv_bfloat16* dst, int ld, const float (&a)[N], int nt, int lane) {
  const uint32_t sel = lane & 1 ? 0x3276u : 0x5410u;
  const bool b1 = lane & 2;
  uint32_t x[N / 2];      // two features of token 2 u + (lane & 1)
#pragma unroll
  for (int u = 0; u < N / 2; ++u) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a[2 * u], a[2 * u + 1]);
    x[u] = *reinterpret_cast<const uint32_t*>(&h);
  }
#pragma unroll
  for (int u = 0; u < N / 2; ++u) x[u] = __byte_perm(x[u], __shfl_xor_sync(0xffffffffu, x[u], 1), sel);
  uint2 o[N / 4];         // four features of token 4 s + (lane & 3)
#pragma unroll
  for (int s = 0; s < N / 4; ++s) {
    const uint32_t r = __shfl_xor_sync(0xffffffffu, b1 ? x[2 * s] : x[2 * s + 1], 2);
    o[s] = b1 ? make_uint2(r, x[2 * s + 1]) : make_uint2(x[2 * s], r);
  }
  char* row = reinterpret_cast<char*>(dst + (long long)(lane & 3) * ld + (lane >> 2) * 4);
  const long long step = 8ll * ld;
  if (nt >= N) {          // warp-uniform
#pragma unroll
    for (int s = 0; s < N / 4; ++s) *reinterpret_cast<uint2*>(row + s * step) = o[s];
  } else {
    const int left = nt - (lane & 3);
#pragma unroll
    for (int s = 0; s < N / 4; ++s)
      if (4 * s < left) *reinterpret_cast<uint2*>(row + s * step) = o[s];
  }
}

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The fields that both forms take over as they are.
static inline void fill_params(GemmParams& p, const FfnArgs& a) {
  p.act[0] = static_cast<__nv_bfloat16*>(a.act); p.act[1] = static_cast<__nv_bfloat16*>(a.act_sh);
  p.x = static_cast<const __nv_bfloat16*>(a.x); p.ld_x = a.d->hidden;
  p.row_token = a.row_token; p.row_gate = a.row_gate; p.acc = a.acc;
  p.y[0] = a.y; p.y[1] = a.ysh; p.deterministic = a.deterministic;
  p.yb[0] = static_cast<__nv_bfloat16*>(a.yb); p.yb[1] = static_cast<__nv_bfloat16*>(a.ybsh); p.pair = a.pair;
  p.status = a.d_status;
  p.wscale[0][0][0] = a.w->w_gate_scale; p.wscale[0][0][1] = a.w->w_up_scale;
  p.wscale[0][1][0] = a.w->ws_gate_scale; p.wscale[0][1][1] = a.w->ws_up_scale;
  p.wscale[1][0][0] = p.wscale[1][0][1] = a.w->w_down_scale;
  p.wscale[1][1][0] = p.wscale[1][1][1] = a.w->ws_down_scale;
}

// bf16 row-major [rows, cols] tensor, box = 64 columns x box_rows rows, 128-byte swizzle.
static inline bool make_map(fmmoe_handle* h, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  if (rows == 0) rows = 1;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 2};
  const cuuint32_t box[2] = {64, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = reinterpret_cast<EncodeTiledFn>(h->encode_tiled)(
      m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}


// FP8 bytes, row-major [rows, cols], box = 64 bytes x box_rows rows, no swizzle (read by threads, not by the MMA).
static inline bool make_map_u8(fmmoe_handle* h, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  if (rows == 0) rows = 1;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols};
  const cuuint32_t box[2] = {64, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = reinterpret_cast<EncodeTiledFn>(h->encode_tiled)(
      m, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(base), dims, strides, box, estr,
      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

}  // namespace fmmoe
