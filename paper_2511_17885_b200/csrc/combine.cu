// Last step of Eq. 4: turn the fp32 combine result into the layer output.
// Atomic mode: the GEMM-2 epilogue has already summed g_j * FFN_j(x) and the shared
// experts into `acc`; this kernel adds the residual (optional) and rounds to the
// storage type (fp32 without the residual: `acc` is the output, and this kernel does not run).  Deterministic mode: the per-pair outputs y were stored instead and
// are summed here in a fixed order (slots 0..K-1, then shared experts 0..N_s-1).
#include <cuda_bf16.h>

#include "internal.h"
#include "ptx.cuh"

namespace fmmoe {

struct FinalizeDev {
  const void* x; void* out; long long T; int H, K, n_shared, add_residual, deterministic;
  const float* acc; const float* y; const float* ysh; const int32_t* inv_row; const float* topk_w;
  const __nv_bfloat16* yb; const __nv_bfloat16* ybsh;
};

// the same sums for one 8-column piece of one token: rows rows[0..KK-1] in slot order, shared experts, residual; rounded
template <int KK, bool EARLY>
__device__ __forceinline__ uint4 finalize_piece(const FinalizeDev& a, long long t, int c, const int (&rows)[KK]);

__device__ __forceinline__ void add_bf16x8(float (&v)[8], const uint4 u) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
    v[2 * i] += f.x; v[2 * i + 1] += f.y;
  }
}

// Pair-row mode (bf16 layers, large batches): GEMM-2 wrote every pair's gate-scaled output row once, in bf16.
// out[t] = sum over the token's slots 0..K-1 (its rows through inv_row), then the shared experts 0..N_s-1,
// then the residual, in that fixed order in fp32; one rounding to bf16.  No atomics anywhere, so the result is
// reproducible bit for bit.  A thread owns 8 neighbouring columns of one token: the rows' 16-byte pieces are
// independent loads.
template <int KK, bool EARLY>
__device__ __forceinline__ uint4 finalize_piece(const FinalizeDev& a, long long t, int c, const int (&rows)[KK]) {
  // EARLY: every load before the first sum, what does not depend on `rows` (the residual, up to two shared experts) first, then the
  // row pieces; without it the shared rows and the residual each wait for the sum before them.  Not in the pruning form, which
  // has no registers left for it (80 -> 85 us on 14,336 tokens).
  const bool early_x = EARLY && a.add_residual, s0 = EARLY && a.n_shared > 0, s1 = EARLY && a.n_shared > 1;
  uint4 q[KK], qx = make_uint4(0u, 0u, 0u, 0u), q0 = qx, q1 = qx;
  if (early_x) qx = *reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(a.x) + t * a.H + c);
  if (s0) q0 = *reinterpret_cast<const uint4*>(a.ybsh + t * a.H + c);
  if (s1) q1 = *reinterpret_cast<const uint4*>(a.ybsh + (a.T + t) * a.H + c);
#pragma unroll
  for (int s = 0; s < KK; ++s)      // a padded slot (-1) reads row 0 and is not added
    q[s] = *reinterpret_cast<const uint4*>(a.yb + (long long)(rows[s] < 0 ? 0 : rows[s]) * a.H + c);
  float v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = 0.f;
#pragma unroll
  for (int s = 0; s < KK; ++s)
    if (rows[s] >= 0) add_bf16x8(v, q[s]);
  if (s0) add_bf16x8(v, q0);
  if (s1) add_bf16x8(v, q1);
  for (int s = EARLY ? 2 : 0; s < a.n_shared; ++s)
    add_bf16x8(v, *reinterpret_cast<const uint4*>(a.ybsh + ((long long)s * a.T + t) * a.H + c));
  if (early_x) add_bf16x8(v, qx);
  else if (a.add_residual) add_bf16x8(v, *reinterpret_cast<const uint4*>(static_cast<const __nv_bfloat16*>(a.x) + t * a.H + c));
  uint32_t w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat162 h2 = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    w[j] = *reinterpret_cast<const uint32_t*>(&h2);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// One merged window by one CTA: the members' output rows as finalize_piece gives them (their own blocks store them), their
// mean rescaled to the largest member norm (Eq. 16-18) from the rounded rows, with the sums in compact_kernel's order.
// A thread owns 8 columns: rows of at most 2,048.
template <int KK>
__device__ __forceinline__ void finalize_merged_window(const FinalizeDev& a, const FinalizePrune& pr, int k0) {
  constexpr int MAXW = FMMOE_MAX_WINDOW;
  __shared__ float s_red[8][MAXW + 1];
  __shared__ int s_rows[MAXW][KK];
  __shared__ int s_tok[MAXW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int b = 0;
  while (b + 1 < pr.sq.n_seq && k0 >= pr.sq.m[b]) { k0 -= pr.sq.m[b]; ++b; }
  const int2 e = pr.merges[pr.sq.win_off[b] + k0];
  if (e.x < pr.sq.out_off[b] || e.x >= pr.sq.out_off[b + 1]) return;   // open entry: inconsistent mask / count (status word set)
  const int v0 = e.y < 0 || e.y + pr.W > pr.sq.n_vis[b] ? 0 : e.y;     // same: stay inside the list
  const long long s_lo = pr.sq.seq_off[b], s_hi = pr.sq.seq_off[b + 1];
  for (int i = tid; i < pr.W * KK; i += 256) {
    const int k = i / KK;
    int t = pr.vis_list[s_lo + v0 + k];
    if (t < s_lo || t >= s_hi) t = (int)s_lo;
    if (i == k * KK) s_tok[k] = t;
    s_rows[k][i - k * KK] = a.inv_row[(long long)t * KK + i - k * KK];
  }
  __syncthreads();
  const bool on = tid < a.H / 8;
  float part[MAXW + 1], mean[8];
#pragma unroll
  for (int k = 0; k <= MAXW; ++k) part[k] = 0.f;
#pragma unroll
  for (int j = 0; j < 8; ++j) mean[j] = 0.f;
  const float invW = 1.f / (float)pr.W;
  if (on) {
#pragma unroll
    for (int k = 0; k < MAXW; ++k) {
      if (k < pr.W) {
        int rows[KK];
#pragma unroll
        for (int s = 0; s < KK; ++s) rows[s] = s_rows[k][s];
        const uint4 q = finalize_piece<KK, false>(a, s_tok[k], tid * 8, rows);
        float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        add_bf16x8(f, q);
#pragma unroll
        for (int j = 0; j < 8; ++j) { part[k] = fmaf(f[j], f[j], part[k]); mean[j] += f[j]; }
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) { const float mv = mean[j] * invW; part[MAXW] = fmaf(mv, mv, part[MAXW]); }
  }
#pragma unroll
  for (int k = 0; k <= MAXW; ++k) {
    if (k < pr.W || k == MAXW) {
#pragma unroll
      for (int o = 16; o; o >>= 1) part[k] += __shfl_xor_sync(0xffffffffu, part[k], o);
      if (lane == 0) s_red[warp][k] = part[k];
    }
  }
  __syncthreads();
  float nmax = 0.f, nb = 0.f;
#pragma unroll
  for (int k = 0; k <= MAXW; ++k) {
    if (k < pr.W || k == MAXW) {
      float tot = 0.f;
#pragma unroll
      for (int ww = 0; ww < 8; ++ww) tot += s_red[ww][k];
      if (k < MAXW) nmax = fmaxf(nmax, sqrtf(tot)); else nb = sqrtf(tot);
    }
  }
  const float scale = (pr.merge_mode == 1 ? 1.f : (nb > 0.f ? nmax / nb : 0.f)) * invW;   // Eq. 18
  if (on) {
    uint32_t w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const __nv_bfloat162 h2 = __floats2bfloat162_rn(mean[2 * j] * scale, mean[2 * j + 1] * scale);
      w[j] = *reinterpret_cast<const uint32_t*>(&h2);
    }
    *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(pr.x_out) + (long long)e.x * a.H + tid * 8) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// PRUNE: the call's pruning stage is done here too (fmmoe_moe_forward_prune): a token that is kept stores its row twice, and
// the first CTAs form the merged windows.  That takes the place of a pass that reads the layer output back from L2 and
// of its launch: 20.7 us against 18.8 + 8.3 us on 3,584 tokens, 65 against 59 + 21 us on 14,336.  The merged windows' members
// are summed a second time (3-11 % of the tokens), in front, because theirs is the longest chain.
template <int KK, bool PRUNE>
__device__ __forceinline__ void finalize_pair_body(const FinalizeDev& a, const FinalizePrune* pr) {
  pdl_launch_dependents();
  pdl_wait();
  const int n_merges = PRUNE ? pr->n_merges : 0;
  if (PRUNE && (int)blockIdx.x < n_merges) {
    finalize_merged_window<KK>(a, *pr, (int)blockIdx.x);
    return;
  }
  const unsigned hv = a.H / 8;
  const unsigned long long n = (unsigned long long)a.T * hv, step = (unsigned long long)((int)gridDim.x - n_merges) * 256;
  for (unsigned long long i = (unsigned long long)((int)blockIdx.x - n_merges) * 256 + threadIdx.x; i < n; i += step) {
    // a piece: a token and 8 columns (a 64-bit division for each would be a third of the instructions)
    const unsigned long long t64 = n >> 32 ? i / hv : (unsigned)i / hv;
    const long long t = (long long)t64;
    const int c = (int)(i - t64 * hv) * 8;
    int rows[KK];
#pragma unroll
    for (int s = 0; s < KK; ++s) rows[s] = a.inv_row[t * KK + s];
    const int pos = PRUNE ? pr->pos[t] : -1;
    const uint4 v = finalize_piece<KK, !PRUNE>(a, t, c, rows);
    *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(a.out) + t * a.H + c) = v;
    if (PRUNE && pos >= 0) *reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(pr->x_out) + (long long)pos * a.H + c) = v;
  }
}
template <int KK>
__global__ void __launch_bounds__(256) finalize_pair_kernel(const FinalizeDev a) { finalize_pair_body<KK, false>(a, nullptr); }
template <int KK>
__global__ void __launch_bounds__(256) finalize_pair_prune_kernel(const FinalizeDev a, const __grid_constant__ FinalizePrune pr) {
  finalize_pair_body<KK, true>(a, &pr);
}

template <int KK>
static cudaError_t launch_finalize_pair(const FinalizeDev& d, const FinalizePrune* pr, unsigned blocks, cudaStream_t s) {
  if (pr) return launch_pdl(finalize_pair_prune_kernel<KK>, dim3(blocks + (unsigned)pr->n_merges), dim3(256), 0, s, 1, d, *pr);
  return launch_pdl(finalize_pair_kernel<KK>, dim3(blocks), dim3(256), 0, s, 1, d);
}
typedef cudaError_t (*FinalizePairFn)(const FinalizeDev&, const FinalizePrune*, unsigned, cudaStream_t);
static const FinalizePairFn kFinalizePair[FMMOE_MAX_TOPK] = {
    launch_finalize_pair<1>,  launch_finalize_pair<2>,  launch_finalize_pair<3>,  launch_finalize_pair<4>,
    launch_finalize_pair<5>,  launch_finalize_pair<6>,  launch_finalize_pair<7>,  launch_finalize_pair<8>,
    launch_finalize_pair<9>,  launch_finalize_pair<10>, launch_finalize_pair<11>, launch_finalize_pair<12>,
    launch_finalize_pair<13>, launch_finalize_pair<14>, launch_finalize_pair<15>, launch_finalize_pair<16>};

template <typename T> struct Vec4;
template <> struct Vec4<float> {
  static __device__ __forceinline__ float4 load(const float* p) { return *reinterpret_cast<const float4*>(p); }
  static __device__ __forceinline__ void store(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
};
template <> struct Vec4<__nv_bfloat16> {
  static __device__ __forceinline__ float4 load(const __nv_bfloat16* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
  }
  static __device__ __forceinline__ void store(__nv_bfloat16* p, float4 v) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    uint2 u;
    u.x = *reinterpret_cast<const uint32_t*>(&a);
    u.y = *reinterpret_cast<const uint32_t*>(&b);
    *reinterpret_cast<uint2*>(p) = u;
  }
};

template <typename T>
__global__ void finalize_kernel(const FinalizeDev a) {
  pdl_launch_dependents();
  pdl_wait();
  const int hv = a.H / 4;
  const long long n = a.T * hv;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const long long t = i / hv;
    const int c = (int)(i - t * hv) * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (!a.deterministic) {
      v = *reinterpret_cast<const float4*>(a.acc + t * a.H + c);
    } else {
      for (int s = 0; s < a.K; ++s) {
        const int row = a.inv_row[t * a.K + s];
        if (row < 0) continue;
        const float g = a.topk_w[t * a.K + s];
        const float4 yv = *reinterpret_cast<const float4*>(a.y + (long long)row * a.H + c);
        v.x = fmaf(g, yv.x, v.x); v.y = fmaf(g, yv.y, v.y); v.z = fmaf(g, yv.z, v.z); v.w = fmaf(g, yv.w, v.w);
      }
      for (int s = 0; s < a.n_shared; ++s) {
        const float4 yv = *reinterpret_cast<const float4*>(a.ysh + ((long long)s * a.T + t) * a.H + c);
        v.x += yv.x; v.y += yv.y; v.z += yv.z; v.w += yv.w;
      }
    }
    if (a.add_residual) {
      const float4 xv = Vec4<T>::load(static_cast<const T*>(a.x) + t * a.H + c);
      v.x += xv.x; v.y += xv.y; v.z += xv.z; v.w += xv.w;
    }
    Vec4<T>::store(static_cast<T*>(a.out) + t * a.H + c, v);
  }
}

fmmoe_status launch_finalize(fmmoe_handle* h, const FinalizeArgs& a, cudaStream_t s) {
  if (a.T == 0) return FMMOE_OK;
  FinalizeDev d;
  d.x = a.x; d.out = a.out; d.T = a.T; d.H = a.H; d.K = a.K; d.n_shared = a.n_shared;
  d.add_residual = a.add_residual; d.deterministic = a.deterministic;
  d.acc = a.acc; d.y = a.y; d.ysh = a.ysh; d.inv_row = a.inv_row; d.topk_w = a.topk_w;
  d.yb = static_cast<const __nv_bfloat16*>(a.yb); d.ybsh = static_cast<const __nv_bfloat16*>(a.ybsh);
  if (a.pair) {
    if (a.dtype != FMMOE_BF16 || a.H % 8 || a.K < 1 || a.K > FMMOE_MAX_TOPK || (a.prune && a.H > 2048)) return FMMOE_ERR_INTERNAL;
    const long long n8 = a.T * (a.H / 8);
    long long blocks8 = (n8 + 255) / 256;
    const long long cap8 = (long long)h->sm_count * 32;
    if (blocks8 > cap8) blocks8 = cap8;
    {
      ProfScope ps(h, FMMOE_KERNEL_FINALIZE, s);
      for (int rep = 0; rep < ps.reps; ++rep) {
        FMMOE_CUDA_TRY(kFinalizePair[a.K - 1](d, a.prune, (unsigned)blocks8, s));
        h->launches += 1;
      }
    }
    FMMOE_CUDA_TRY(cudaGetLastError());
    return FMMOE_OK;
  }
  const long long n = a.T * (a.H / 4);
  const int threads = 256;
  long long blocks = (n + threads - 1) / threads;
  const long long cap = (long long)h->sm_count * 16;
  if (blocks > cap) blocks = cap;
  {
    ProfScope ps(h, FMMOE_KERNEL_FINALIZE, s);
    for (int rep = 0; rep < ps.reps; ++rep) {
      if (a.dtype == FMMOE_BF16) FMMOE_CUDA_TRY(launch_pdl(finalize_kernel<__nv_bfloat16>, dim3((unsigned)blocks), dim3(threads), 0, s, 1, d));
      else FMMOE_CUDA_TRY(launch_pdl(finalize_kernel<float>, dim3((unsigned)blocks), dim3(threads), 0, s, 1, d));
      h->launches += 1;
    }
  }
  FMMOE_CUDA_TRY(cudaGetLastError());
  return FMMOE_OK;
}

}  // namespace fmmoe
