// Router: logits (Eq. 1), softmax (Eq. 2), modality-aware top-k (Eq. 3, with K_v
// for vision tokens once the layer has reached l_v) and renormalised gates (Eq. 5),
// fused in one kernel per storage type.
//   bf16: the logits tile [128 tokens, E] is a tcgen05 GEMM fed by TMA with its accumulator
//         in tensor memory; the tile is then copied to shared memory and eight lanes per
//         token run the softmax / top-k / gate step across the expert dimension.
//   fp32: a CTA owns 32 tokens, a warp one or two; it forms their logits with plain FMA from shared memory (TF32
//         would miss an fp32 tolerance) and runs the softmax / top-k / gate step across the expert dimension with
//         warp shuffles.
// Both kernels also start the permutation: a CTA records, per expert, which of its tokens
// selected it (a bit mask in shared memory), from which it writes the block's expert counts
// and, for every (token, slot), the rank of the token among the block's tokens that chose
// the same expert.  Ranks come from bit counts, never from the arrival order of atomics.
#include <cuda_bf16.h>
#include <float.h>

#include "internal.h"
#include "ptx.cuh"

namespace fmmoe {

constexpr int R_BM = 32;
constexpr int R_BK = 64;            // k elements per slab of the fp32 router
constexpr int R_LD = R_BK + 4;      // its row pitch: 16-byte reads of eight rows hit distinct banks

struct RouteDev {
  const void* x; const void* w; const float* bias; const uint8_t* is_visual;
  long long T; int H, E, K, Kv, reduce_on, e_pad;
  float* logits; float* probs; int32_t* topk_idx; float* topk_w; int32_t* inv_row;
  int32_t* blk_cnt; int ld_blk;  // [E][ld_blk] selections of each token block per expert
  float* acc_zero; int32_t* misc_zero;   // combine accumulator [T,H] / scheduler words to clear (or NULL)
  long long misc_ints;
  // the whole permutation in this kernel (all CTAs are one cluster): outputs of permute.cu's kernels
  int fuse, block_m;
  int32_t* expert_off; int32_t* row_token; float* row_gate; MTile* mtiles; int32_t* n_mtiles;
  unsigned long long wait_budget_ns;     // time budget of every bounded wait
  int* status;
  int test_cta, test_k_block;            // self-test: this CTA's producer stops before this k-block (-1: its wait for the peers' counts runs out)
};

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Softmax / top-k / gates for the CTA's tokens, logits already in shared memory.
// NTL = e_pad / 32 values per lane.
template <int NTL>
__device__ __forceinline__ void route_tail(const float* Ls, int ldl, long long t0, const RouteDev& a, uint32_t* emask, int* s_topk, float* s_topw) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int r = warp; r < R_BM; r += blockDim.x >> 5) {
    const long long t = t0 + r;
    if (t >= a.T) break;
    float v[NTL];
#pragma unroll
    for (int j = 0; j < NTL; ++j) {
      const int e = lane + 32 * j;
      v[j] = e < a.E ? Ls[r * ldl + e] : -INFINITY;
    }
    if (a.logits) {
#pragma unroll
      for (int j = 0; j < NTL; ++j)
        if (lane + 32 * j < a.E) a.logits[t * a.E + lane + 32 * j] = v[j];
    }
    // The shuffle reductions below need a total order: non-finite logits (overflowed activations
    // upstream) are clamped and NaN counts as the lowest value, so that all lanes agree on every
    // round's winner and each selected index is a valid, distinct expert.  Finite inputs are untouched.
#pragma unroll
    for (int j = 0; j < NTL; ++j)
      if (lane + 32 * j < a.E) v[j] = fminf(fmaxf(v[j], -FLT_MAX), FLT_MAX);
    float m = v[0];
#pragma unroll
    for (int j = 1; j < NTL; ++j) m = fmaxf(m, v[j]);
    m = warp_max(m);
    float s = 0.f;
#pragma unroll
    for (int j = 0; j < NTL; ++j) s += expf(v[j] - m);   // exp(-inf) = 0 for padded lanes
    s = warp_sum(s);
    if (a.probs) {
      const float inv = 1.f / s;
#pragma unroll
      for (int j = 0; j < NTL; ++j)
        if (lane + 32 * j < a.E) a.probs[t * a.E + lane + 32 * j] = expf(v[j] - m) * inv;
    }
    const int k_t = (a.reduce_on && a.is_visual[t]) ? a.Kv : a.K;
    uint32_t taken = 0;
    float my_val = -INFINITY;
    int my_idx = -1;
    for (int i = 0; i < k_t; ++i) {
      float bv = -INFINITY;
      int be = 0x7fffffff;
#pragma unroll
      for (int j = 0; j < NTL; ++j) {
        const int e = lane + 32 * j;
        if (e < a.E && !((taken >> j) & 1u) && (v[j] > bv || be == 0x7fffffff)) { bv = v[j]; be = e; }
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
        const int oe = __shfl_xor_sync(0xffffffffu, be, o);
        if (oe != 0x7fffffff && (be == 0x7fffffff || ov > bv || (ov == bv && oe < be))) { bv = ov; be = oe; }
      }
      if ((be & 31) == lane) taken |= 1u << (be >> 5);
      if (lane == i) { my_val = bv; my_idx = be; }
    }
    const float p = lane < k_t ? expf(my_val - m) : 0.f;
    const float denom = warp_sum(p);
    if (lane < a.K) {
      const bool sel = lane < k_t;
      const float wgt = sel ? p / denom : 0.f;
      a.topk_idx[t * a.K + lane] = s_topk[r * a.K + lane] = sel ? my_idx : -1;
      a.topk_w[t * a.K + lane] = s_topw[r * a.K + lane] = wgt;
      if (sel && (unsigned)my_idx < (unsigned)a.E) atomicOr(&emask[my_idx], 1u << r);   // one 32-bit word per expert: the block has 32 tokens
    }
  }
}

// After the block's selections are in `emask` ([E][WORDS] bit masks over the block's tokens):
// write the block's per-expert counts and the in-block rank of every (token, slot).
// `s_topk`: the block's selections in shared memory.
template <int WORDS>
__device__ __forceinline__ void emit_block_ranks(const uint32_t* emask, const int* s_topk, long long t0, int blk, const RouteDev& a) {
  __syncthreads();
  for (int e = threadIdx.x; e < a.E; e += blockDim.x) {
    int c = 0;
#pragma unroll
    for (int w = 0; w < WORDS; ++w) c += __popc(emask[e * WORDS + w]);
    a.blk_cnt[(long long)e * a.ld_blk + blk] = c;
  }
  const int items = WORDS * 32 * a.K;
  for (int it = threadIdx.x; it < items; it += blockDim.x) {
    const int r = it / a.K;
    const long long t = t0 + r;
    if (t >= a.T) break;
    const int e = s_topk[it];
    int rank = -1;
    if (e >= 0 && e < a.E) {
      rank = __popc(emask[e * WORDS + (r >> 5)] & ((1u << (r & 31)) - 1u));
#pragma unroll
      for (int w = 0; w < WORDS; ++w)
        if (w < (r >> 5)) rank += __popc(emask[e * WORDS + w]);
    }
    a.inv_row[t * a.K + (it - r * a.K)] = rank;
  }
}

// ---------------------------------------------------------------------------------------
// bf16 router on the tcgen05 tensor cores.  A CTA of 16 warps owns 128 tokens:
//   warp 0    : TMA producer  (X tile 128x64 and the router matrix tile e_pad x 64 per stage)
//   warp 1    : UMMA issuer   (128 x e_pad x 16 tcgen05.mma; the logits tile lives in TMEM)
//   warps 4-11: once the accumulator is complete, copy it from TMEM to shared memory, reusing the pipeline's
//               stage buffers
//   cluster   : with few token tiles the contraction is split over a cluster of 2 or 4 CTAs
//               (more SMs pulling X); every CTA then owns 128/split rows of the tile and adds
//               the partial rows of its peers, in rank order: each peer pushes them by a bulk copy that signals the
//               owner's barrier, where shared memory has room for them, or is read by the owner (4 % off one token of the 64-expert layer, 1 % off 16 tokens of the
//               128-expert layer, together with the counts below, the late cluster wait and a producer that does not wait for
//               the mask; from 200 tokens on no difference beyond the noise)
//   all warps : softmax / top-k / gates with 8 lanes per token (4 tokens per warp at a time):
//               every lane holds E/8 logits of its token in registers, the row maximum, the
//               sum and each top-k round are a local scan plus three shuffle steps across
//               the expert dimension.
// The router matrix is read once per 128 tokens (from L2 after the first CTA), X once.
// ---------------------------------------------------------------------------------------
constexpr int RT_BM = 128;
constexpr int RT_BK = 64;
constexpr int RT_THREADS = 512;
constexpr int RT_A_BYTES = RT_BM * RT_BK * 2;
constexpr int RT_MAX_STAGES = 8;

__device__ __forceinline__ float group8_max(float v) {
#pragma unroll
  for (int o = 4; o; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
__device__ __forceinline__ float group8_sum(float v) {
#pragma unroll
  for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ int group8_min_int(int v) {
#pragma unroll
  for (int o = 4; o; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}
template <int NV> __device__ __forceinline__ float tree_max(const float (&z)[NV]) {
  float b[NV];
#pragma unroll
  for (int j = 0; j < NV; ++j) b[j] = z[j];
#pragma unroll
  for (int n = NV; n > 1; n = (n + 1) / 2)
#pragma unroll
    for (int j = 0; j < n / 2; ++j) b[j] = fmaxf(b[j], b[j + (n + 1) / 2]);
  return b[0];
}

// Softmax / top-k / gates for n_rows (a multiple of 32) token rows whose logits (without the bias)
// sit in shared memory, row pitch ldl (odd).  Eight lanes per token, four tokens per warp.
// NV = logits per lane (expert e = lane8 + 8 j), NV * 8 >= E.
// Its time is its instructions: about 950 clocks a round for 128 rows of 128 experts (16 warps).  Other layouts
// measured slower there: sixteen lanes per token 18.4k against 13.0k clocks (32 rows: 7.8k against 7.2k), a warp per token
// with integer warp reductions 33k, a warp per token by bisection on keys with votes 41k, value and index through one tree 18k.
template <int NV>
__device__ __forceinline__ void route_tail_group8(const float* Lr, int ldl, const float* bias_s, long long t_first, int n_rows,
                                                  uint32_t* emask, int words, const uint8_t* s_k, int* s_topk, float* s_topw,
                                                  const RouteDev& a) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 3, l8 = lane & 7;
  const int E = a.E;
#pragma unroll 1
  for (int base = (warp >> 3) * 32; base < n_rows; base += 32 * (RT_THREADS / 256)) {
    // eight warps share 32 rows; rows of one warp are 8 apart: with an odd row pitch the four groups hit
    // distinct banks
    const int rl = base + g * 8 + (warp & 7);
    const long long t = t_first + rl;
    const bool tok_ok = t < a.T;
    float z[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const int e = l8 + 8 * j;
      z[j] = e < E ? Lr[rl * ldl + e] + bias_s[e] : -INFINITY;
    }
    if (a.logits && tok_ok) {
#pragma unroll
      for (int j = 0; j < NV; ++j)
        if (l8 + 8 * j < E) a.logits[t * E + l8 + 8 * j] = z[j];
    }
    // The selection below marks a taken entry with -inf and looks experts up by value, so it needs
    // finite logits: non-finite ones (overflowed activations upstream) are clamped, NaN counts as the
    // lowest value.  Finite inputs are untouched; whatever the input, every selected index is a
    // valid, distinct expert.
#pragma unroll
    for (int j = 0; j < NV; ++j)
      if (l8 + 8 * j < E) z[j] = fminf(fmaxf(z[j], -FLT_MAX), FLT_MAX);
    const float m = group8_max(tree_max(z));
    if (a.probs) {
      float s = 0.f;
#pragma unroll
      for (int j = 0; j < NV; ++j) s += __expf(z[j] - m);   // exp(-inf) = 0 for padded entries
      s = group8_sum(s);
      if (tok_ok) {
        const float inv = 1.f / s;
#pragma unroll
        for (int j = 0; j < NV; ++j)
          if (l8 + 8 * j < E) a.probs[t * E + l8 + 8 * j] = __expf(z[j] - m) * inv;
      }
    }
    const int k_t = s_k[rl];
    const int k_warp = __reduce_max_sync(0xffffffffu, k_t);
    float denom = 0.f;
    float sel_p[2] = {0.f, 0.f};
    int sel_e[2] = {-1, -1};
    float bv = m;
#pragma unroll 1
    for (int i = 0; i < k_warp; ++i) {
      // largest remaining logit of the token, then the lowest expert index that holds it
      // (a taken entry is overwritten with -inf; real logits are finite)
      if (i) bv = group8_max(tree_max(z));
      int be = 0x7fffffff;
#pragma unroll
      for (int j = NV - 1; j >= 0; --j)
        if (z[j] == bv) be = l8 + 8 * j;
      be = group8_min_int(be);
      if (i < k_t) {
#pragma unroll
        for (int j = 0; j < NV; ++j)
          if (l8 + 8 * j == be) z[j] = -INFINITY;
        const float p = __expf(bv - m);
        denom += p;
        if ((i & 7) == l8) { if (i < 8) { sel_p[0] = p; sel_e[0] = be; } else { sel_p[1] = p; sel_e[1] = be; } }
      }
    }
    if (tok_ok) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int slot = l8 + 8 * h;
        if (slot < a.K) {
          const bool sel = slot < k_t;
          const int idx = sel ? sel_e[h] : -1;
          const float wgt = sel ? sel_p[h] / denom : 0.f;            // Eq. 5
          a.topk_idx[t * a.K + slot] = idx;
          a.topk_w[t * a.K + slot] = wgt;
          s_topk[rl * a.K + slot] = idx;
          s_topw[rl * a.K + slot] = wgt;
          if (sel && (unsigned)idx < (unsigned)E) atomicOr(&emask[idx * words + (rl >> 5)], 1u << (rl & 31));
        }
      }
    }
  }
}

// The whole permutation for a batch whose router CTAs form one cluster (see launch_route_tc): with every CTA's per-expert
// counts at hand (s_all [CTA][E], pushed by its peers) a CTA derives the rows of its own pairs and writes them;
// CTA 0 writes the expert offsets and the M-tile list.  The same stable order as permute.cu, without its two kernels:
// at these sizes each of them is a launch and a few dependent loads (5-8 and 5-6 us) in front of GEMM-1.
// s_tmp: [3 * FMMOE_MAX_EXPERTS + 64] ints of shared memory.
__device__ __forceinline__ void permute_in_cluster(const int* s_all, const uint32_t* emask, int words, const int* s_topk, const float* s_topw,
                                                   long long t_first, int n_rows, int* s_tmp, const RouteDev& a) {
  int* s_base = s_tmp;                             // [E] row of this CTA's first pair of the expert
  int* s_cnt = s_tmp + FMMOE_MAX_EXPERTS;          // [E] rows of the expert
  int* s_off = s_tmp + 2 * FMMOE_MAX_EXPERTS;      // [E] first row of the expert
  int* s_wsum = s_tmp + 3 * FMMOE_MAX_EXPERTS;     // [2][8] sums of 32 experts: rows, M-tiles
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)blockIdx.x, n_cta = (int)gridDim.x;
  int cnt = 0, before = 0, nt = 0, ic = 0, it = 0;
  if (tid < FMMOE_MAX_EXPERTS) {                   // eight warps, an expert per thread
    if (tid < a.E) {
      for (int q = 0; q < n_cta; ++q) {
        const int c = s_all[q * a.E + tid];
        if (q < rank) before += c;
        cnt += c;
      }
    }
    nt = (cnt + a.block_m - 1) / a.block_m;
    ic = cnt; it = nt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n1 = __shfl_up_sync(0xffffffffu, ic, o), n2 = __shfl_up_sync(0xffffffffu, it, o);
      if (lane >= o) { ic += n1; it += n2; }
    }
    if (lane == 31) { s_wsum[warp] = ic; s_wsum[8 + warp] = it; }
  }
  __syncthreads();
  if (tid < FMMOE_MAX_EXPERTS) {
    int row0 = ic - cnt, tile0 = it - nt;
    for (int w = 0; w < warp; ++w) { row0 += s_wsum[w]; tile0 += s_wsum[8 + w]; }
    if (tid < a.E) {
      s_base[tid] = row0 + before;
      s_cnt[tid] = cnt; s_off[tid] = row0;
      if (rank == 0) {
        a.expert_off[tid] = row0;
        if (tid == a.E - 1) { a.expert_off[a.E] = row0 + cnt; a.n_mtiles[0] = tile0 + nt; }
        const int bm = mtile_rows(cnt, nt, a.block_m);
        for (int i = 0; i < nt; ++i) {
          MTile m;
          m.group = tid; m.row0 = row0 + i * bm;
          m.rows = min(bm, cnt - i * bm); m.pad = nt == 1;
          a.mtiles[tile0 + i] = m;
        }
      }
    }
  }
  __syncthreads();
  for (int i = tid; i < n_rows * a.K; i += (int)blockDim.x) {
    const int r = i / a.K;
    const long long t = t_first + r;
    if (t >= a.T) break;
    const int e = s_topk[i];
    int row = -1;
    if (e >= 0 && e < a.E) {
      row = s_base[e] + __popc(emask[e * words + (r >> 5)] & ((1u << (r & 31)) - 1u));
      for (int w = 0; w < (r >> 5); ++w) row += __popc(emask[e * words + w]);
      if (row < s_off[e] + s_cnt[e]) {             // always, for a consistent record
        a.row_token[row] = (int32_t)t;
        a.row_gate[row] = s_topw[i];
      }
    }
    a.inv_row[t * a.K + (i - r * a.K)] = row;
  }
}

// What a CTA whose wait ran out leaves: the kernels behind the router take rows and tokens from the routing record, so its
// tokens read as having selected nothing, and its block has no counts (emask, which a cluster's exchange counts, is still all
// zero), whatever the buffers held before.  No shared memory: a late copy may still land in the stage buffers.
__device__ __forceinline__ void record_nothing(long long t_first, int items, const RouteDev& a) {
  for (int i = threadIdx.x; i < items; i += blockDim.x) {
    const long long t = t_first + i / a.K, p = t * a.K + i % a.K;
    if (t < a.T) { a.topk_idx[p] = -1; a.topk_w[p] = 0.f; a.inv_row[p] = -1; }
  }
  if (!a.fuse)
    for (int e = threadIdx.x; e < a.E; e += blockDim.x) a.blk_cnt[(long long)e * a.ld_blk + blockIdx.x] = 0;
}

// Behind the tail of a router whose CTAs are one cluster: every CTA's counts go to every other, then the permutation.  `failed`: this
// CTA gave up before (its emask is all zero).  Ends with this CTA's arrival at the cluster's last barrier.
__device__ __forceinline__ void exchange_and_permute(int* s_all, uint64_t* cnt_bar, volatile int* peer_gave_up, const uint32_t* emask, int words,
                                                     const int* s_topk, const float* s_topw, long long t_first, int n_rows, int* s_tmp,
                                                     unsigned long long budget, bool clustered, bool& failed, const RouteDev& a) {
  for (int i = threadIdx.x; i < (int)gridDim.x * a.E; i += blockDim.x) {      // this CTA's counts to every CTA
    const int q = i / a.E, e = i - q * a.E;
    int c = 0;
    for (int w = 0; w < words; ++w) c += __popc(emask[e * words + w]);
    int* dst = s_all + (int)blockIdx.x * a.E + e;
    if (q == (int)blockIdx.x) *dst = c;
    else st_async_u32(cluster_map_shared(smem_u32(dst), (uint32_t)q), (uint32_t)c, cluster_map_shared(smem_u32(cnt_bar), (uint32_t)q));
  }
  // Stores that signal the receiver's barrier: a cluster barrier here would first wait for the tail's writes to global memory
  // (1,800-4,500 clocks).
  const bool ok = mbar_wait_cluster(cnt_bar, 0, nullptr, budget) && !((int)blockIdx.x == a.test_cta && a.test_k_block < 0);
  // Its peers have counted this CTA's pairs, whose rows will now not be written: CTA 0 takes the record back
  if (!ok) {
    st_cluster_u32(cluster_map_shared(smem_u32(const_cast<int*>(peer_gave_up)), 0), 1u);
    cluster_fence();
  }
  if (clustered) cluster_arrive_relaxed();
  if (__syncthreads_or(!ok) && !failed) {
    failed = true;
    if (threadIdx.x == 0) atomicCAS(a.status, 0, DEV_TIMEOUT);
    record_nothing(t_first, n_rows * a.K, a);
  }
  if (!failed) permute_in_cluster(s_all, emask, words, s_topk, s_topw, t_first, n_rows, s_tmp, a);
}

__global__ void __launch_bounds__(RT_THREADS, 1)
route_tc_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW, const RouteDev a,
                const int stages, const int tmem_cols, const int tile_bytes, const int recv_bytes, const int split, int* status) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  unsigned char* smem = smem_raw + ((1024 - (raw & 1023)) & 1023);
  const int b_bytes = a.e_pad * RT_BK * 2;
  const int stage_bytes = RT_A_BYTES + b_bytes;
  float* recv = reinterpret_cast<float*>(smem + tile_bytes);                // push: [split - 1][n_rows][ldl] the peers' partial rows
  float* bias_s = reinterpret_cast<float*>(smem + tile_bytes + recv_bytes); // [256]
  uint32_t* emask = reinterpret_cast<uint32_t*>(bias_s + FMMOE_MAX_EXPERTS);   // [256][4] token masks per expert
  const int row_items = RT_BM / split * a.K;
  int* s_topk = reinterpret_cast<int*>(emask + FMMOE_MAX_EXPERTS * 4);       // [128 / split][K] selections of this CTA's tokens
  float* s_topw = reinterpret_cast<float*>(s_topk + row_items);              // and their gates
  uint8_t* s_k = reinterpret_cast<uint8_t*>(s_topw + row_items);             // [128] experts each of this CTA's tokens takes
  int* s_all = reinterpret_cast<int*>(s_k + RT_BM);                          // a.fuse: [CTA][E] selections per expert
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(s_all + (a.fuse ? (((int)gridDim.x * a.E + 1) & ~1) : 0));   // row_items is a multiple of 32
  uint64_t* empty_bar = full_bar + RT_MAX_STAGES;
  uint64_t* tfull_bar = empty_bar + RT_MAX_STAGES;
  uint64_t* rx_bar = tfull_bar + 1;      // push: the peers' partial rows have arrived
  uint64_t* cnt_bar = rx_bar + 1;        // a.fuse: every CTA's counts have arrived
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(cnt_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* peer_gave_up = abort_flag + 1;   // a.fuse, in CTA 0: a peer that had sent its counts then gave up
  const int warp = warp_index(), lane = threadIdx.x & 31;
  // this CTA's slice of the contraction (a cluster is one tile's CTAs, or with a.fuse all CTAs of the grid)
  const int krank = (int)blockIdx.x % split;
  const int crank0 = (int)cluster_ctarank() - krank;   // cluster rank of the tile's first CTA
  const int kblocks = a.H / RT_BK / split;
  const int kb0 = krank * kblocks;
  const int nch = (a.E + 31) / 32;
  const int n_rows = RT_BM / split, row_lo = krank * n_rows, words = n_rows / 32;   // the tile rows this CTA owns
  const int ldl = nch * 32 + 1;                 // odd pitch of the logits tile in shared memory
  float* Ls = reinterpret_cast<float*>(smem);   // [128][ldl] (partial) logits, overlays the stage buffers after the GEMM
  float* Lr = Ls + row_lo * ldl;                // [n_rows][ldl] this CTA's rows, completed in place (32 odd-pitch rows: 128-byte aligned)
  const bool clustered = split > 1 || (a.fuse && gridDim.x > 1);      // a single CTA is launched without a cluster
  // rows of the tile that CTA q of it owns and that exist
  auto valid_rows = [&](int q) {
    const long long left = a.T - ((long long)(blockIdx.x / split) * RT_BM + q * n_rows);
    return left < 0 ? 0 : left < n_rows ? (int)left : n_rows;
  };
  auto slab_bytes = [&](int rows) { return (uint32_t)(rows * ldl * 4 + 15) & ~15u; };

  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; ++i) { mbar_init(&full_bar[i], 1); mbar_init(&empty_bar[i], 1); }
    mbar_init(tfull_bar, 1);
    mbar_init(rx_bar, 1); mbar_init(cnt_bar, 1);
    *abort_flag = 0; *peer_gave_up = 0;
    mbar_fence_init();
    if (recv_bytes) mbar_arrive_expect_tx(rx_bar, (uint32_t)(split - 1) * slab_bytes(valid_rows(krank)));
    if (a.fuse) mbar_arrive_expect_tx(cnt_bar, (gridDim.x - 1) * (uint32_t)a.E * 4u);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, (uint32_t)tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // "this CTA runs and its barriers exist": waited for before anything is sent to a peer, behind the GEMM
  if (clustered) cluster_arrive();
  // The router matrix may have left L2 since the last layer: ask for this CTA's slice before the predecessor is done.
  // (A prefetch into L2, the point of coherence: harmless even if the predecessor were to write the matrix.)
  if (threadIdx.x == 0 && (int)blockIdx.x < 2 * split) {
    for (int kb = 0; kb < kblocks; ++kb) tma_prefetch_l2_2d(&tmW, (kb0 + kb) * RT_BK, 0);
  }
  pdl_wait();   // from here on: global memory that earlier kernels of the stream may have written
  // The successor may start from here on.  Not before the wait, nor before the tile schedulers' counters are cleared: the expert
  // GEMMs' small-M form starts on shared experts beside the router, and takes what is in front of the layer as done.
  if (blockIdx.x != 0) {
    pdl_launch_dependents();
  } else if (warp == 3) {
    if (a.misc_zero)
      for (long long i = 1 + lane; i < a.misc_ints; i += 32) a.misc_zero[i] = 0;
    __threadfence();
    __syncwarp();
    pdl_launch_dependents();
  }
  const int row0 = (blockIdx.x / split) * RT_BM;

  if (warp == 0) {
    if (elect_one()) {
      tma_prefetch_desc(&tmX); tma_prefetch_desc(&tmW);
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      // self-test: the issuer's wait for the first stage left out runs out
      const int kb_end = (int)blockIdx.x == a.test_cta && a.test_k_block >= 0 ? min(a.test_k_block, kblocks) : kblocks;
      for (int kb = 0; kb < kb_end; ++kb) {
        if (!mbar_wait(&empty_bar[stage], phase ^ 1, abort_flag, a.wait_budget_ns)) { ok = false; break; }
        unsigned char* sA = smem + stage * stage_bytes;
        mbar_arrive_expect_tx(&full_bar[stage], (uint32_t)stage_bytes);
        tma_load_2d(sA, &tmX, &full_bar[stage], (kb0 + kb) * RT_BK, row0);
        tma_load_2d(sA + RT_A_BYTES, &tmW, &full_bar[stage], (kb0 + kb) * RT_BK, 0);
        if (++stage == stages) { stage = 0; phase ^= 1; }
      }
      if (!ok) { atomicCAS(status, 0, DEV_TIMEOUT); *abort_flag = 1; }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      const uint32_t idesc = umma_idesc_bf16(RT_BM, a.e_pad);
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      for (int kb = 0; kb < kblocks; ++kb) {
        if (!mbar_wait(&full_bar[stage], phase, abort_flag, a.wait_budget_ns)) { ok = false; break; }
        tc_fence_after();
        const uint32_t sA = smem_u32(smem + stage * stage_bytes);
        const uint64_t da = umma_desc_sw128(sA);
        const uint64_t db = umma_desc_sw128(sA + RT_A_BYTES);
#pragma unroll
        for (int k = 0; k < RT_BK / 16; ++k) umma_bf16(tmem_base, da + 2 * k, db + 2 * k, idesc, (kb | k) != 0);
        umma_commit(&empty_bar[stage]);
        if (++stage == stages) { stage = 0; phase ^= 1; }
      }
      if (ok) umma_commit(tfull_bar);
      else { atomicCAS(status, 0, DEV_TIMEOUT); *abort_flag = 1; }
    }
  } else {
    // warps 2-15 have nothing to do while the GEMM streams: the modality mask and the bias (behind the GEMM their loads would be a round trip to memory by themselves; nothing of it is in front of the producer),
    // this CTA's rows of the layer's fp32 combine accumulator
    if (threadIdx.x >= RT_THREADS - RT_BM) {
      const int r = threadIdx.x - (RT_THREADS - RT_BM);
      const long long t = (long long)row0 + row_lo + r;
      if (r < n_rows) s_k[r] = (uint8_t)(t < a.T ? ((a.reduce_on && a.is_visual[t]) ? a.Kv : a.K) : 0);
    }
    for (int e = threadIdx.x - 64; e < FMMOE_MAX_EXPERTS; e += RT_THREADS - 64) {
      bias_s[e] = (a.bias && e < a.E) ? a.bias[e] : 0.f;
#pragma unroll
      for (int w = 0; w < 4; ++w) emask[e * 4 + w] = 0;
    }
    if (a.acc_zero) {
      const int n_rows = RT_BM / split;
      const long long t_lo = (long long)row0 + krank * n_rows;
      long long t_hi = t_lo + n_rows;
      if (t_hi > a.T) t_hi = a.T;
      if (t_lo < t_hi) {
        float4* dst = reinterpret_cast<float4*>(a.acc_zero + t_lo * a.H);
        const long long n4 = (t_hi - t_lo) * a.H / 4;
        for (long long i = threadIdx.x - 64; i < n4; i += RT_THREADS - 64) dst[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  }
  if (clustered) cluster_wait();      // every CTA of the cluster runs: 1,300-1,900 clocks, most warps pass them while the GEMM streams
  if (warp >= 4 && warp < 12) {
    // accumulator complete => every stage buffer has been consumed: reuse them for the logits
    // (two warps per TMEM lane quarter, alternate 32-column chunks)
    const int q = warp & 3;
    if (mbar_wait_warp(tfull_bar, 0, abort_flag, a.wait_budget_ns)) {
      tc_fence_after();
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
      float* dst = Ls + (q * 32 + lane) * ldl;
      const bool any = (long long)row0 + q * 32 < a.T;      // some of the quarter's rows exist
      for (int c = (warp - 4) >> 2; any && c < nch; c += 2) {
        uint32_t v[32];
        tmem_ld32(taddr + c * 32, v);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 32; ++j) dst[c * 32 + j] = __uint_as_float(v[j]);   // this CTA's partial sums
      }
      if (recv_bytes) fence_proxy_async_smem();      // read by bulk copies
    } else {
      atomicCAS(status, 0, DEV_TIMEOUT); *abort_flag = 1;
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  bool failed = *abort_flag != 0;
  if (failed) {
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 200000ull) { }
    __syncthreads();
  }
  // What peers wait for is sent unconditionally (a CTA that gave up sends what its buffers hold), and every CTA passes the same
  // cluster barriers, so no peer can be left waiting.
  const unsigned long long peer_budget = 2 * a.wait_budget_ns + 1000000ull;      // a peer may first have to give up a wait of its own
  if (recv_bytes) {
    // Every CTA of the tile gets its rows of this CTA's partial tile (those that exist) by one bulk copy that signals its
    // barrier, and adds them up in rank order.  Against reading the peers' tiles behind a cluster barrier, whose release and
    // acquire alone took 2,600-3,500 clocks and the reads 1,900-3,300.
    if (warp == 0 && elect_one()) {
      for (int q = 0; q < split; ++q) {
        const uint32_t bytes = slab_bytes(valid_rows(q));
        if (q == krank || bytes == 0) continue;
        const int slot = krank < q ? krank : krank - 1;
        bulk_copy_to_cluster(cluster_map_shared(smem_u32(recv + slot * n_rows * ldl), (uint32_t)(crank0 + q)), smem_u32(Ls + q * n_rows * ldl),
                             bytes, cluster_map_shared(smem_u32(rx_bar), (uint32_t)(crank0 + q)));
      }
    }
    const bool ok = mbar_wait(rx_bar, 0, nullptr, peer_budget);
    const int n4 = (int)(slab_bytes(valid_rows(krank)) >> 4);
    for (int i = threadIdx.x; i < n4; i += RT_THREADS) {
      float4 own = reinterpret_cast<float4*>(Lr)[i], sum;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (q >= split) break;
        const float4 v = q == krank ? own : reinterpret_cast<const float4*>(recv + (q < krank ? q : q - 1) * n_rows * ldl)[i];
        if (q == 0) sum = v;
        else { sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w; }
      }
      reinterpret_cast<float4*>(Lr)[i] = sum;
    }
    // The CTA's rows are here; it stays until its peers have theirs (the wait is at the end of the kernel)
    if (!a.fuse) cluster_arrive_relaxed();
    if (__syncthreads_or(!ok) && !failed) {
      failed = true;
      if (threadIdx.x == 0) { atomicCAS(status, 0, DEV_TIMEOUT); *abort_flag = 1; }
    }
  } else if (split > 1) {
    // no room to receive: read the peers' rows
    cluster_sync_all();   // every CTA of the tile holds its partial logits in shared memory
    if (!failed) {
      // This CTA's rows of the logits tile = sum over the cluster's partial tiles, in rank order.
      // The rows are one contiguous, 16-byte aligned run of every CTA's tile
      // (32 rows * pitch * 4 bytes), read from the peers with 16-byte distributed-shared-memory loads.
      uint32_t peer[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) peer[q] = cluster_map_shared(smem_u32(Lr), (uint32_t)(crank0 + (q < split ? q : 0)));
      const int n4 = n_rows * ldl / 4;
      for (int i = threadIdx.x; i < n4; i += RT_THREADS) {
        float4 p[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < split) p[q] = ld_cluster_v4f32(peer[q] + i * 16);
#pragma unroll
        for (int q = 1; q < 4; ++q)
          if (q < split) { p[0].x += p[q].x; p[0].y += p[q].y; p[0].z += p[q].z; p[0].w += p[q].w; }
        reinterpret_cast<float4*>(Lr)[i] = p[0];
      }
    }
    if (!a.fuse) cluster_arrive_relaxed();
    __syncthreads();
  }
  const long long t_first = (long long)row0 + row_lo;
  if (!failed) {
    switch (nch) {
      case 1: route_tail_group8<4>(Lr, ldl, bias_s, t_first, n_rows, emask, words, s_k, s_topk, s_topw, a); break;
      case 2: route_tail_group8<8>(Lr, ldl, bias_s, t_first, n_rows, emask, words, s_k, s_topk, s_topw, a); break;
      case 3: route_tail_group8<12>(Lr, ldl, bias_s, t_first, n_rows, emask, words, s_k, s_topk, s_topw, a); break;
      case 4: route_tail_group8<16>(Lr, ldl, bias_s, t_first, n_rows, emask, words, s_k, s_topk, s_topw, a); break;
      case 5: route_tail_group8<20>(Lr, ldl, bias_s, t_first, n_rows, emask, words, s_k, s_topk, s_topw, a); break;
      case 6: route_tail_group8<24>(Lr, ldl, bias_s, t_first, n_rows, emask, words, s_k, s_topk, s_topw, a); break;
      case 7: route_tail_group8<28>(Lr, ldl, bias_s, t_first, n_rows, emask, words, s_k, s_topk, s_topw, a); break;
      default: route_tail_group8<32>(Lr, ldl, bias_s, t_first, n_rows, emask, words, s_k, s_topk, s_topw, a); break;
    }
    __syncthreads();
    // the token block of this CTA: rows [row_lo, row_lo + n_rows) of the tile
    if (!a.fuse) {
      if (split == 1) emit_block_ranks<4>(emask, s_topk, t_first, blockIdx.x, a);
      else if (split == 2) emit_block_ranks<2>(emask, s_topk, t_first, blockIdx.x, a);
      else emit_block_ranks<1>(emask, s_topk, t_first, blockIdx.x, a);
    }
  } else {
    record_nothing(t_first, row_items, a);
  }
  if (a.fuse)
    exchange_and_permute(s_all, cnt_bar, peer_gave_up, emask, words, s_topk, s_topw, t_first, n_rows, reinterpret_cast<int*>(Lr), peer_budget, clustered, failed, a);
  if (clustered) cluster_wait();   // peers may still be reading this CTA's tile until here
  if (failed && clustered) {       // what they sent before may still be under way to a CTA that no longer waits for it
    const uint64_t t0 = global_timer_ns();
    while (global_timer_ns() - t0 < 200000ull) { }
  }
  __syncthreads();
  if (a.fuse && blockIdx.x == 0 && (failed || *peer_gave_up)) {   // a wait ran out: leave the expert GEMMs no tiles to follow
    for (int e = threadIdx.x; e <= a.E; e += RT_THREADS) a.expert_off[e] = 0;
    if (threadIdx.x == 0) a.n_mtiles[0] = 0;
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, (uint32_t)tmem_cols);
  }
}

// fp32 router (no tensor cores: TF32 would miss the fp32 tolerance).  A CTA owns 32 tokens, a warp TPW of them, lane l experts l,
// l+32, ...; X and W_E come in slabs of 64 k by cp.async, up to four of them on their way, and are read as 16-byte vectors.  A CTA's time is
// its latency (8 CTAs at 256 tokens): of the slabs, of the tail and, up to eight CTAs, of the exchange of counts that spares the permutation's kernel.
// TPW: one token a warp (1,024 threads) up to 16 experts, where the lanes share the contraction and the tail counts; beyond, two (512 threads): what bounds
// it then is the rows of W_E read from shared memory, which serve both, and a thread has 128 registers (with 64 the kernels for more than 96 experts
// spill).  With the permutation, in a graph, one / two tokens a warp: H 256, 8 experts: 256 tokens 8.2 / 8.2 us, 4,096 tokens 10.1 / 10.3; 32 experts: 256 tokens
// 15.2 / 13.9; H 2,048, 4,096 tokens: 32 experts 71.9 / 54.9, 128 experts 181.7 / 119.1, 256 experts 332.9 / 201.0.  (H 2,048 and 8 experts, which nothing
// here is made for, would be faster with two as well: 30.5 / 25.9.)
template <int NT> struct RouteF32 {
  static constexpr int E_PAD = NT * 32, LDL = E_PAD + 1, STAGES = NT <= 2 ? 4 : 2;
  static constexpr int SLAB = (R_BM + E_PAD) * R_LD;              // floats: [R_BM rows of X | E_PAD rows of W_E][R_LD]
  static constexpr int TMP = 3 * FMMOE_MAX_EXPERTS + 64;          // ints of permute_in_cluster, over the slabs
  static constexpr int SLABS = STAGES * SLAB > TMP ? STAGES * SLAB : TMP;
  static size_t bytes(int E, int K, int n_cta) {                  // + logits, emask, selections, gates, counts
    return 4 * ((size_t)SLABS + R_BM * LDL + E_PAD + 2 * R_BM * K + (size_t)n_cta * E);
  }
};
template <int NT, int TPW>
__global__ void __launch_bounds__(R_BM * 32 / TPW, 1) route_f32_kernel(const RouteDev a) {
  constexpr int R_THREADS = R_BM * 32 / TPW, WARPS = R_BM / TPW;      // warp w: tokens w, w + WARPS
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint64_t cnt_bar;             // a.fuse: every CTA's counts have arrived
  __shared__ int peer_gave_up;             // a.fuse, in CTA 0: a peer that had sent its counts then gave up
  using L = RouteF32<NT>;
  float* slabs = reinterpret_cast<float*>(smem_raw);
  float* Ls = slabs + L::SLABS;                                     // [R_BM][LDL]
  uint32_t* emask = reinterpret_cast<uint32_t*>(Ls + R_BM * L::LDL);   // [E_PAD] one word per expert (32 tokens)
  int* s_topk = reinterpret_cast<int*>(emask + L::E_PAD);           // [R_BM][K]
  float* s_topw = reinterpret_cast<float*>(s_topk + R_BM * a.K);
  int* s_all = reinterpret_cast<int*>(s_topw + R_BM * a.K);         // a.fuse: [CTA][E] selections per expert
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long t0 = (long long)blockIdx.x * R_BM;
  const bool clustered = a.fuse && gridDim.x > 1;      // a single CTA is launched without a cluster
  pdl_launch_dependents();
  if (a.fuse) {
    if (tid == 0) {
      mbar_init(&cnt_bar, 1);
      peer_gave_up = 0;
      mbar_fence_init();
      mbar_arrive_expect_tx(&cnt_bar, (gridDim.x - 1) * (uint32_t)a.E * 4u);
    }
    __syncthreads();
    if (clustered) cluster_arrive();      // "this CTA runs and its barrier exists": waited for before anything is sent
  }
  pdl_wait();
  if (a.misc_zero && blockIdx.x == 0)
    for (long long i = 1 + tid; i < a.misc_ints; i += R_THREADS) a.misc_zero[i] = 0;
  const float* X = static_cast<const float*>(a.x);
  const float* W = static_cast<const float*>(a.w);
  const uint32_t smem0 = smem_u32(slabs);
  const int n_slabs = (a.H + R_BK - 1) / R_BK;
  auto load_slab = [&](int s) {                      // a group of its own, also where there is none left
    constexpr int PR = R_BK / 4;                     // 16-byte pieces per row
    const int k0 = s * R_BK, stage = s % L::STAGES;
    if (s < n_slabs)
      for (int c = tid; c < (R_BM + a.E) * PR; c += R_THREADS) {   // rows of experts that do not exist stay as they are
        const int r = c / PR, k = k0 + c % PR * 4;
        const bool is_x = r < R_BM;
        const bool ok = k < a.H && (!is_x || t0 + r < a.T);        // H is a multiple of 4
        const float* src = is_x ? X + (t0 + r) * a.H + k : W + (long long)(r - R_BM) * a.H + k;
        cp_async_16_or_zero(smem0 + 4u * (uint32_t)(stage * L::SLAB + r * R_LD + c % PR * 4), ok ? src : X, ok);
      }
    cp_async_commit();
  };
#pragma unroll
  for (int s = 0; s < L::STAGES; ++s) load_slab(s);
  if (a.acc_zero) {   // clear this block's rows of the combine accumulator
    long long t_hi = t0 + R_BM;
    if (t_hi > a.T) t_hi = a.T;
    float4* dst = reinterpret_cast<float4*>(a.acc_zero + t0 * a.H);
    const long long n = (t_hi - t0) * a.H / 4;
    for (long long i = tid; i < n; i += R_THREADS) dst[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  for (int i = tid; i < L::E_PAD; i += R_THREADS) emask[i] = 0;
  // Few experts: the lanes that would hold none take their share of the contraction, four or two k-quadruples a step
  const int ks = TPW > 1 || a.E > 16 ? 1 : a.E > 8 ? 2 : 4, e_lane = lane & (32 / ks - 1), k_lane = lane / (32 / ks) * 4;
  float2 acc[TPW][NT];
  float bias[NT];
#pragma unroll
  for (int i = 0; i < TPW; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll
  for (int j = 0; j < NT; ++j) { bias[j] = a.bias && lane + 32 * j < a.E ? a.bias[lane + 32 * j] : 0.f; }
  for (int s = 0; s < n_slabs; ++s) {
    cp_async_wait_all_but<L::STAGES - 1>();
    __syncthreads();
    const float* Xs = slabs + (s % L::STAGES) * L::SLAB + warp * R_LD + k_lane;
    const float* Ws = slabs + (s % L::STAGES) * L::SLAB + (R_BM + e_lane) * R_LD + k_lane;
#pragma unroll 2
    for (int k = 0; k < R_BK; k += 4 * ks) {
      float4 xv[TPW], wv[NT];
#pragma unroll
      for (int i = 0; i < TPW; ++i) xv[i] = *reinterpret_cast<const float4*>(Xs + i * WARPS * R_LD + k);
#pragma unroll
      for (int j = 0; j < NT; ++j) wv[j] = *reinterpret_cast<const float4*>(Ws + 32 * j * R_LD + k);
#pragma unroll
      for (int i = 0; i < TPW; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j) {
          fma2(acc[i][j], make_float2(xv[i].x, xv[i].y), make_float2(wv[j].x, wv[j].y));
          fma2(acc[i][j], make_float2(xv[i].z, xv[i].w), make_float2(wv[j].z, wv[j].w));
        }
    }
    __syncthreads();
    load_slab(s + L::STAGES);
  }
#pragma unroll
  for (int i = 0; i < TPW; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j) {
      float z = acc[i][j].x + acc[i][j].y;
      if (ks == 4) z += __shfl_xor_sync(0xffffffffu, z, 8);
      if (ks > 1) z += __shfl_xor_sync(0xffffffffu, z, 16);
      if (lane < 32 / ks) Ls[(warp + i * WARPS) * L::LDL + lane + 32 * j] = z + bias[j];
    }
  __syncwarp();       // a warp reads its own tokens' rows
  route_tail<NT>(Ls, L::LDL, t0, a, emask, s_topk, s_topw);
  if (!a.fuse) {
    emit_block_ranks<1>(emask, s_topk, t0, blockIdx.x, a);
    return;
  }
  __syncthreads();
  if (clustered) cluster_wait();
  bool failed = false;
  exchange_and_permute(s_all, &cnt_bar, &peer_gave_up, emask, 1, s_topk, s_topw, t0, R_BM, reinterpret_cast<int*>(slabs), a.wait_budget_ns, clustered, failed, a);
  if (clustered) cluster_wait();   // peers may still be sending to this CTA until here
  if (failed && clustered) {       // what they sent before may still be under way to a CTA that no longer waits for it
    const uint64_t t1 = global_timer_ns();
    while (global_timer_ns() - t1 < 200000ull) { }
  }
  __syncthreads();
  if (blockIdx.x == 0 && (failed || *(volatile int*)&peer_gave_up)) {   // a wait ran out: leave the expert GEMMs no tiles to follow
    for (int e = tid; e <= a.E; e += R_THREADS) a.expert_off[e] = 0;
    if (tid == 0) a.n_mtiles[0] = 0;
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static bool route_map(fmmoe_handle* h, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {cols * 2};
  const cuuint32_t box[2] = {RT_BK, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return reinterpret_cast<EncodeTiledFn>(h->encode_tiled)(
             m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

static fmmoe_status launch_route_tc(fmmoe_handle* h, RouteDev d, cudaStream_t s) {
  if (!h->encode_tiled) return FMMOE_ERR_CUDA;
  d.e_pad = (d.E + 15) / 16 * 16;                       // UMMA N: a multiple of 16 for M = 128
  const int stage_bytes = RT_A_BYTES + d.e_pad * RT_BK * 2;
  const int split = route_split(d.T, d.H);
  const int n_cta = (int)((d.T + RT_BM - 1) / RT_BM) * split;
  const size_t extra = FMMOE_MAX_EXPERTS * 20 + (size_t)RT_BM / split * d.K * 8 + RT_BM + (d.fuse ? ((size_t)n_cta * d.E + 1) / 2 * 8 : 0) +
                       (2 * RT_MAX_STAGES + 3) * 8 + 16 + 1024;
  const size_t row_bytes = (size_t)((d.E + 31) / 32 * 32 + 1) * 4, logit_bytes = (RT_BM * row_bytes + 1023) / 1024 * 1024;
  const int kblocks = d.H / RT_BK / split;
  auto ring_stages = [&](size_t recv) {
    const int room = h->max_smem_optin - (int)(extra + recv), most = kblocks < RT_MAX_STAGES ? kblocks : RT_MAX_STAGES;
    const int n = (room < 200 * 1024 ? room : 200 * 1024) / stage_bytes;
    return n < most ? n : most;
  };
  // Room for the peers' partial rows beside the CTA's own tile, if there is any (a split of four: up to 224 experts), and if it leaves
  // the ring four stages (up to 160 experts) or there are at most half a tile's rows to send.  The router alone (H 2,048, top-8), rows
  // pushed / read, us: 128 experts, 1 token 9.6 / 11.4, 64 tokens 11.8 / 12.3, 2,432 tokens (five stages of six) 12.5 / 12.1; 192
  // experts, 64 tokens 15.0 / 15.3, 128 tokens 15.9 / 15.4, 2,432 tokens (three of five) 16.4 / 15.3; 224 experts, 64 tokens 16.9 / 16.5,
  // 2,432 tokens 18.0 / 16.5.  Inside a layer the difference is small: 128 experts, 686 tokens 222.1 / 222.7, 3,584 tokens 287.8 /
  // 290.0; 192 experts of 384 features, 2,432 tokens 184.7 / 185.0; 224 experts, 256 tokens 181.8 / 181.1, 2,432 tokens 206.3 / 206.8.
  size_t recv_bytes = (size_t)(split - 1) * (RT_BM / split) * row_bytes;
  if (logit_bytes + recv_bytes + extra > (size_t)h->max_smem_optin || (d.T > RT_BM / 2 && ring_stages(recv_bytes) < 4 && ring_stages(recv_bytes) < ring_stages(0)))
    recv_bytes = 0;
  const int stages = ring_stages(recv_bytes);
  if (stages < 1) return FMMOE_ERR_UNSUPPORTED;
  int tmem_cols = 32;
  while (tmem_cols < (d.E + 31) / 32 * 32) tmem_cols *= 2;
  // the logits tile, [128][32*ceil(E/32)+1] fp32, overlays the stage buffers
  size_t tile_bytes = (size_t)stages * stage_bytes;
  if (logit_bytes > tile_bytes) tile_bytes = logit_bytes;
  const size_t smem = tile_bytes + recv_bytes + extra;
  CUtensorMap mx, mw;
  if (!route_map(h, &mx, d.x, (uint64_t)d.T, (uint64_t)d.H, RT_BM)) return FMMOE_ERR_CUDA;
  if (!route_map(h, &mw, d.w, (uint64_t)d.E, (uint64_t)d.H, (uint32_t)d.e_pad)) return FMMOE_ERR_CUDA;
  if (!h->route_attr_set) {   // once per handle: the largest size any shape can ask for
    FMMOE_CUDA_TRY(cudaFuncSetAttribute(route_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, h->max_smem_optin));
    h->route_attr_set = true;
  }
  if (smem > (size_t)h->max_smem_optin) return FMMOE_ERR_UNSUPPORTED;
  const int tiles = (int)((d.T + RT_BM - 1) / RT_BM);
  {
    ProfScope ps(h, FMMOE_KERNEL_ROUTE, s);
    for (int rep = 0; rep < ps.reps; ++rep) {
      FMMOE_CUDA_TRY(launch_pdl(route_tc_kernel, dim3((unsigned)(tiles * split)), dim3(RT_THREADS), smem, s, (unsigned)(d.fuse ? tiles * split : split), mx, mw, d,
                                stages, tmem_cols, (int)tile_bytes, (int)recv_bytes, split, h->d_status));
      h->launches += 1;
    }
  }
  FMMOE_CUDA_TRY(cudaGetLastError());
  return FMMOE_OK;
}

template <int NT, int TPW = 2>
static fmmoe_status launch_nt(fmmoe_handle* h, const RouteDev& d, int grid, cudaStream_t s) {
  constexpr uint32_t bit = 1u << (TPW == 1 ? 0 : NT);
  const size_t smem = RouteF32<NT>::bytes(d.E, d.K, d.fuse ? grid : 0);
  if (!(h->route_f32_attr_mask & bit)) {      // once per handle: what any shape can ask for
    FMMOE_CUDA_TRY(cudaFuncSetAttribute(route_f32_kernel<NT, TPW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)RouteF32<NT>::bytes(NT * 32, FMMOE_MAX_TOPK, 8)));
    h->route_f32_attr_mask |= bit;
  }
  {
    ProfScope ps(h, FMMOE_KERNEL_ROUTE, s);
    for (int rep = 0; rep < ps.reps; ++rep) {
      FMMOE_CUDA_TRY(launch_pdl(route_f32_kernel<NT, TPW>, dim3(grid), dim3(R_BM * 32 / TPW), smem, s, (unsigned)(d.fuse ? grid : 1), d));
      h->launches += 1;
    }
  }
  FMMOE_CUDA_TRY(cudaGetLastError());
  return FMMOE_OK;
}

fmmoe_status launch_route(fmmoe_handle* h, const RouteArgs& a, cudaStream_t s) {
  if (a.T == 0) return FMMOE_OK;
  RouteDev d;
  d.x = a.x; d.w = a.router_w; d.bias = a.router_b; d.is_visual = a.is_visual;
  d.T = a.T; d.H = a.H; d.E = a.E; d.K = a.K; d.Kv = a.Kv; d.reduce_on = a.reduce_on;
  d.e_pad = (a.E + 31) / 32 * 32;
  d.logits = a.logits; d.probs = a.probs; d.topk_idx = a.topk_idx; d.topk_w = a.topk_w;
  d.inv_row = a.inv_row; d.blk_cnt = a.blk_cnt; d.acc_zero = a.acc_zero; d.misc_zero = a.misc_zero; d.misc_ints = a.misc_ints;
  d.ld_blk = route_blk_stride(a.dtype, a.T, a.H);
  d.fuse = a.fuse; d.block_m = a.block_m;
  d.expert_off = a.expert_off; d.row_token = a.row_token; d.row_gate = a.row_gate; d.mtiles = a.mtiles; d.n_mtiles = a.n_mtiles;
  fmmoe_status st;
  d.wait_budget_ns = h->wait_budget_ns; d.status = h->d_status; d.test_cta = -1; d.test_k_block = 0;
  if (h->test_route_cta >= 0 && (a.dtype == FMMOE_BF16 || (a.fuse && h->test_route_k_block < 0))) {     // armed self-test: this call only
    d.test_cta = h->test_route_cta; d.test_k_block = h->test_route_k_block; d.wait_budget_ns = h->test_route_budget_ns;
    h->test_route_cta = -1;
  }
  if (a.dtype == FMMOE_BF16) {
    st = launch_route_tc(h, d, s);
  } else {
    const int grid = (int)((a.T + R_BM - 1) / R_BM);
    switch (d.e_pad / 32) {
      case 1: st = d.E <= 16 ? launch_nt<1, 1>(h, d, grid, s) : launch_nt<1>(h, d, grid, s); break;
      case 2: st = launch_nt<2>(h, d, grid, s); break;
      case 3: st = launch_nt<3>(h, d, grid, s); break;
      case 4: st = launch_nt<4>(h, d, grid, s); break;
      case 5: st = launch_nt<5>(h, d, grid, s); break;
      case 6: st = launch_nt<6>(h, d, grid, s); break;
      case 7: st = launch_nt<7>(h, d, grid, s); break;
      case 8: st = launch_nt<8>(h, d, grid, s); break;
      default: return FMMOE_ERR_UNSUPPORTED;
    }
  }
  return st;
}

}  // namespace fmmoe
