// Permute-by-expert: the stable grouping of the routed (token, expert) pairs by expert.  The
// paper only states that an unselected expert costs nothing (Section 3.1); the grouped order
// used here is the unique stable one (rows of an expert ascend by token index), so it is
// reproducible bit for bit: every rank comes from counts and scans, never from the arrival
// order of atomics.
//
// The router leaves, per block of tokens, the number of selections of every expert (blk_cnt)
// and, per (token, slot), the token's rank among its block's tokens that chose that expert.
//   permute_kernel : up to PB_MAX token blocks: every CTA sums the count table for itself (it is small: 57 KB for 3,584
//                    tokens and 128 experts) and writes the rows of its own block's pairs; CTA 0 also writes expert_off and
//                    the M-tile list.  Beyond, where the table times the CTAs would be too much to read, three steps:
//   scan_kernel    : per expert an exclusive scan of the block counts (in place), the scan of
//                    the expert totals (expert_off) and the list of 128-row M-tiles
//   scatter_kernel : row = expert_off[e] + block offset + in-block rank, for every pair
#include <cuda_bf16.h>

#include "internal.h"
#include "ptx.cuh"

namespace fmmoe {

constexpr int P_THREADS = 1024;

struct PermuteDev {
  const int32_t* topk_idx; const float* topk_w;
  int32_t* blk_cnt; int n_blk, ld_blk, blk_tokens;
  long long T; int K, E, block_m;
  int32_t* expert_off; int32_t* row_token; float* row_gate; int32_t* inv_row;
  MTile* mtiles; int32_t* n_mtiles;
};

// A launch and its dependent loads are what this costs: one kernel, 5.1-5.5 us on 686..3,584 tokens (9.2 us on 19,456), against 8.3 + 4.5 us
// (6.5 + 4.7 us) for scan_kernel and scatter_kernel with a wait between them.  Sums of at most 32,768 tokens: two 16-bit halves of a word
// go through one shuffle reduction.
constexpr int PB_MAX = 256;
constexpr int PB_THREADS = 512;
constexpr int PB_ITEMS = 4;          // pairs per thread: blocks of 128 tokens, 16 slots
// EVEN: an expert's tiles share its rows (CTA pairs).  A form of its own, since the division, where nothing needs it, cost 0.2 us of
// the fp32 layer's 56.
template <bool EVEN>
__global__ void __launch_bounds__(PB_THREADS) permute_kernel(const PermuteDev a) {
  __shared__ uint32_t s_sum[FMMOE_MAX_EXPERTS];                 // rows of the expert | rows before this block << 16
  __shared__ int s_row[FMMOE_MAX_EXPERTS];                      // row of this block's first pair of the expert
  __shared__ int s_wsum[2][FMMOE_MAX_EXPERTS / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, blk = blockIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  // this block's pairs: loads first
  const long long p0 = (long long)blk * a.blk_tokens * a.K;
  const long long left = a.T * a.K - p0;
  const int n_items = left < (long long)a.blk_tokens * a.K ? (int)(left < 0 ? 0 : left) : a.blk_tokens * a.K;
  int e[PB_ITEMS], rank[PB_ITEMS];
  float gate[PB_ITEMS];
#pragma unroll
  for (int u = 0; u < PB_ITEMS; ++u) {
    const int i = tid + u * PB_THREADS;
    e[u] = -1; rank[u] = 0; gate[u] = 0.f;
    if (i < n_items) { e[u] = a.topk_idx[p0 + i]; rank[u] = a.inv_row[p0 + i]; gate[u] = a.topk_w[p0 + i]; }
  }
  // column sums of the count table: four blocks a lane in one 16-byte load, eight experts of a warp in flight
  constexpr int WARPS = PB_THREADS / 32, EX = 8;
  for (int e0 = warp; e0 < a.E; e0 += EX * WARPS) {
    uint32_t acc[EX];
#pragma unroll
    for (int u = 0; u < EX; ++u) acc[u] = 0u;
    for (int b = lane * 4; b < a.n_blk; b += 128) {
      uint4 v[EX];
#pragma unroll
      for (int u = 0; u < EX; ++u)
        if (e0 + u * WARPS < a.E) v[u] = *reinterpret_cast<const uint4*>(a.blk_cnt + (long long)(e0 + u * WARPS) * a.ld_blk + b);
#pragma unroll
      for (int u = 0; u < EX; ++u) {
        if (e0 + u * WARPS >= a.E) break;
        const uint32_t c[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (b + j < a.n_blk) acc[u] += b + j < blk ? c[j] | c[j] << 16 : c[j];
      }
    }
#pragma unroll
    for (int u = 0; u < EX; ++u) {
#pragma unroll
      for (int o = 16; o; o >>= 1) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], o);
      if (lane == 0 && e0 + u * WARPS < a.E) s_sum[e0 + u * WARPS] = acc[u];
    }
  }
  __syncthreads();
  int cnt = 0, nt = 0, ic = 0, it = 0;
  if (tid < FMMOE_MAX_EXPERTS) {      // first row and first M-tile of each expert: an expert per thread
    cnt = tid < a.E ? (int)(s_sum[tid] & 0xffffu) : 0;
    nt = (cnt + a.block_m - 1) / a.block_m;
    ic = cnt; it = nt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int n1 = __shfl_up_sync(0xffffffffu, ic, o), n2 = __shfl_up_sync(0xffffffffu, it, o);
      if (lane >= o) { ic += n1; it += n2; }
    }
    if (lane == 31) { s_wsum[0][warp] = ic; s_wsum[1][warp] = it; }
  }
  __syncthreads();
  if (tid < a.E) {
    int row0 = ic - cnt, tile0 = it - nt;
    for (int w = 0; w < warp; ++w) { row0 += s_wsum[0][w]; tile0 += s_wsum[1][w]; }
    s_row[tid] = row0 + (int)(s_sum[tid] >> 16);
    if (blk == 0) {
      a.expert_off[tid] = row0;
      if (tid == a.E - 1) {
        a.expert_off[a.E] = row0 + cnt;
        if (a.n_mtiles) a.n_mtiles[0] = tile0 + nt;
      }
      if (a.mtiles) {
        const int bm = EVEN ? mtile_rows(cnt, nt, a.block_m) : a.block_m;
        for (int i = 0; i < nt; ++i) {
          MTile m;
          m.group = tid; m.row0 = row0 + i * bm;
          m.rows = min(bm, cnt - i * bm); m.pad = nt == 1;   // 1: the expert's only tile
          a.mtiles[tile0 + i] = m;
        }
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < PB_ITEMS; ++u) {
    if (e[u] < 0 || e[u] >= a.E) continue;              // padded slot: inv_row already holds -1
    const int row = s_row[e[u]] + rank[u];
    if (row < 0 || row >= a.T * a.K) continue;          // cannot happen for a consistent routing record
    const long long p = p0 + tid + u * PB_THREADS;
    a.row_token[row] = (int32_t)(p / a.K);
    a.row_gate[row] = gate[u];
    a.inv_row[p] = row;
  }
}

template <bool EVEN>
__global__ void __launch_bounds__(P_THREADS) scan_kernel(const PermuteDev a) {
  __shared__ int s_cnt[FMMOE_MAX_EXPERTS], s_off[FMMOE_MAX_EXPERTS + 1], s_tile0[FMMOE_MAX_EXPERTS + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_launch_dependents();
  pdl_wait();
  // per expert: exclusive scan over the token blocks, 32 blocks per step
  for (int e = warp; e < a.E; e += P_THREADS / 32) {
    int32_t* row = a.blk_cnt + (long long)e * a.ld_blk;
    int running = 0;
    for (int b0 = 0; b0 < a.n_blk; b0 += 128) {   // four independent loads per lane, then the scans
      int v[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int b = b0 + 32 * j + lane;
        v[j] = b < a.n_blk ? row[b] : 0;
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int b = b0 + 32 * j + lane;
        int incl = v[j];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int n = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += n;
        }
        if (b < a.n_blk) row[b] = running + incl - v[j];
        running += __shfl_sync(0xffffffffu, incl, 31);
      }
    }
    if (lane == 0) s_cnt[e] = running;
  }
  __syncthreads();
  if (warp == 0) {   // scan over the (<= 256) expert totals: first row and first M-tile of each expert
    int run_rows = 0, run_tiles = 0;
    for (int e0 = 0; e0 < a.E; e0 += 32) {
      const int e = e0 + lane;
      const int c = e < a.E ? s_cnt[e] : 0;
      const int nt = (c + a.block_m - 1) / a.block_m;
      int ic = c, it = nt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int n1 = __shfl_up_sync(0xffffffffu, ic, o);
        const int n2 = __shfl_up_sync(0xffffffffu, it, o);
        if (lane >= o) { ic += n1; it += n2; }
      }
      if (e < a.E) { s_off[e] = run_rows + ic - c; s_tile0[e] = run_tiles + it - nt; }
      run_rows += __shfl_sync(0xffffffffu, ic, 31);
      run_tiles += __shfl_sync(0xffffffffu, it, 31);
    }
    if (lane == 0) {
      s_off[a.E] = run_rows; s_tile0[a.E] = run_tiles;
      if (a.n_mtiles) a.n_mtiles[0] = run_tiles;
    }
  }
  __syncthreads();
  for (int e = tid; e <= a.E; e += P_THREADS) a.expert_off[e] = s_off[e];
  if (a.mtiles) {
    for (int e = warp; e < a.E; e += P_THREADS / 32) {
      const int cnt = s_cnt[e], base = s_off[e], nt = s_tile0[e + 1] - s_tile0[e];
      const int bm = EVEN ? mtile_rows(cnt, nt, a.block_m) : a.block_m;
      for (int i = lane; i < nt; i += 32) {
        MTile m;
        m.group = e; m.row0 = base + i * bm;
        m.rows = min(bm, cnt - i * bm); m.pad = nt == 1;   // 1: the expert's only tile
        a.mtiles[s_tile0[e] + i] = m;
      }
    }
  }
}

__global__ void __launch_bounds__(256) scatter_kernel(const PermuteDev a) {
  pdl_launch_dependents();
  pdl_wait();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.T * a.K) return;
  const int e = a.topk_idx[i];
  if (e < 0 || e >= a.E) return;           // padded slot: inv_row already holds -1
  const long long t = i / a.K;
  const int row = a.expert_off[e] + a.blk_cnt[(long long)e * a.ld_blk + (int)(t / a.blk_tokens)] + a.inv_row[i];
  if (row < 0 || row >= a.expert_off[a.E]) return;   // cannot happen for a consistent routing record
  a.row_token[row] = (int32_t)t;
  a.row_gate[row] = a.topk_w[i];
  a.inv_row[i] = row;
}

fmmoe_status launch_permute(fmmoe_handle* h, const PermuteArgs& a, cudaStream_t s) {
  if (a.E <= 0 || a.T <= 0) return FMMOE_OK;
  PermuteDev d;
  d.topk_idx = a.topk_idx; d.topk_w = a.topk_w; d.blk_cnt = a.blk_cnt; d.n_blk = a.n_blk; d.ld_blk = a.ld_blk; d.blk_tokens = a.blk_tokens;
  d.T = a.T; d.K = a.K; d.E = a.E; d.block_m = a.block_m;
  d.expert_off = a.expert_off; d.row_token = a.row_token; d.row_gate = a.row_gate; d.inv_row = a.inv_row;
  d.mtiles = a.mtiles; d.n_mtiles = a.n_mtiles;
  const long long pairs = a.T * a.K;
  {
    ProfScope ps(h, FMMOE_KERNEL_PERMUTE, s);
    if (a.n_blk <= PB_MAX) {
      FMMOE_CUDA_TRY(launch_pdl(a.block_m > TC_BLOCK_M ? permute_kernel<true> : permute_kernel<false>, dim3((unsigned)a.n_blk), dim3(PB_THREADS), 0, s, 1, d));
      FMMOE_CUDA_TRY(cudaGetLastError());
      h->launches += 1;
      return FMMOE_OK;
    }
    FMMOE_CUDA_TRY(launch_pdl(a.block_m > TC_BLOCK_M ? scan_kernel<true> : scan_kernel<false>, dim3(1), dim3(P_THREADS), 0, s, 1, d));
    FMMOE_CUDA_TRY(launch_pdl(scatter_kernel, dim3((unsigned)((pairs + 255) / 256)), dim3(256), 0, s, 1, d));
  }
  FMMOE_CUDA_TRY(cudaGetLastError());
  h->launches += 2;
  return FMMOE_OK;
}

}  // namespace fmmoe
