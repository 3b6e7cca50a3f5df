// Cross-modal attention importance (Eq. 7): the attention weights of the LAST token of every
// sequence (the last text token of [T_v, T_t]) to all tokens, averaged over the attention heads.
// The pruning stage reads the entries at vision tokens (Eq. 11).  Attention layers themselves are
// not part of this library: the caller hands in that layer's keys and the last token's queries.
//
//   logits_kernel  : a CTA per (128 tokens, kv head): dot products of the keys with the queries of the
//                    heads that share this kv head (grouped-query attention), fp32 accumulation; of each head its
//                    tokens' largest logit and their sum of exp below it
//   merge_kernel   : (long sequences, many heads) per sequence and head the softmax's maximum and sum from those of the blocks
//   average_kernel : the same for itself where there was no merge kernel; then a thread per token: mean over heads, in head
//                    order (all in fixed orders: reproducible)
#include <cuda_bf16.h>
#include <math.h>

#include "internal.h"
#include "ptx.cuh"

namespace fmmoe {

constexpr int A_MAXS = FMMOE_MAX_SEQS_PER_LAUNCH;
constexpr int A_MAX_GROUP = 16;   // query heads per kv head
constexpr int A_TOK = 128;        // tokens of a block: every sequence starts a new one
// First block of sequence b (counted over all sequences): its tokens' number of whole blocks and one more for every sequence before it
// hold all of theirs.
__host__ __device__ static inline long long stats_block(long long seq_off, long long b) { return seq_off / A_TOK + b; }
// A maximum to subtract: of nothing but -inf, whose terms are then 0 (a NaN stays one, and the sum with it).
__device__ __forceinline__ float finite_or_zero(float m) { return m == -INFINITY ? 0.f : m; }

struct AttnSeqs {
  int n_seq;
  long long seq_off[A_MAXS + 1];
};

struct AttnDev {
  const void* q; const void* k;
  int n_heads, n_kv, d, group;
  float scale;
  long long T;           // tokens of this launch's sequences start at seq_off[0]
  float* logits;         // [n_heads][T_total]
  float2* stats;         // [block of A_TOK tokens][n_heads] (max, sum exp), a sequence's blocks from stats_block on
  float* out;            // [T_total]
  long long T_total;
  int seq_base;          // index of this launch's first sequence
};

template <typename TT> __device__ __forceinline__ float ld_elem(const TT* p, int i);
template <> __device__ __forceinline__ float ld_elem<float>(const float* p, int i) { return p[i]; }
template <> __device__ __forceinline__ float ld_elem<__nv_bfloat16>(const __nv_bfloat16* p, int i) { return __bfloat162float(p[i]); }

// 16 bytes of a row as fp32 (8 bf16 or 4 fp32 elements)
template <typename TT> struct Piece;
template <> struct Piece<float> {
  static constexpr int N = 4;
  static __device__ __forceinline__ void unpack(const uint4 u, float* f) {
    f[0] = __uint_as_float(u.x); f[1] = __uint_as_float(u.y); f[2] = __uint_as_float(u.z); f[3] = __uint_as_float(u.w);
  }
};
template <> struct Piece<__nv_bfloat16> {
  static constexpr int N = 8;
  static __device__ __forceinline__ void unpack(const uint4 u, float* f) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(w[i] << 16); f[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
  }
};

// Eight lanes share a key: each takes 16-byte pieces l8, l8+8, ... of it, and has four tokens of the CTA in flight,
// so that a query piece (from L1) is converted once for four keys; 128 tokens per CTA.  What bounds it is the latency
// of a round of loads (19,456 tokens with 4 kv heads of 64 are 10 MB of keys: 1.5 us at the memory's rate): 11.3 us
// there, against 67.5 us for a warp per (token, kv head) with its five shuffle steps per head and two-byte loads.
// GM: heads per kv head, rounded up.  VEC = 0: rows that are no multiple of 16 bytes, or pointers that are not aligned.
template <typename TT, int GM, bool VEC>
__global__ void __launch_bounds__(256) attn_logits_kernel(const AttnDev a, const AttnSeqs sq) {
  __shared__ float s_logit[GM][A_TOK];
  pdl_launch_dependents();
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, l8 = lane & 7;
  const int b = blockIdx.y, kvh = (int)(blockIdx.x % (unsigned)a.n_kv);
  const long long t0 = sq.seq_off[b] + (long long)(blockIdx.x / (unsigned)a.n_kv) * A_TOK;
  const int n_tok = (int)min((long long)A_TOK, sq.seq_off[b + 1] - t0);
  if (n_tok <= 0) return;
  const TT* qp = static_cast<const TT*>(a.q) + ((long long)(a.seq_base + b) * a.n_heads + (long long)kvh * a.group) * a.d;
  const int r0 = warp * 4 + (lane >> 3);            // tokens r0, r0 + 32, r0 + 64, r0 + 96 of the block
  const TT* kp[4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
    kp[j] = static_cast<const TT*>(a.k) + ((t0 + min(r0 + 32 * j, n_tok - 1)) * a.n_kv + kvh) * a.d;
  float acc[4][GM];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int g = 0; g < GM; ++g) acc[j][g] = 0.f;
  if (VEC) {
    constexpr int N = Piece<TT>::N;
    for (int i = l8 * N; i < a.d; i += 8 * N) {
      uint4 kq[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) kq[j] = *reinterpret_cast<const uint4*>(kp[j] + i);
      float kf[4][N];
#pragma unroll
      for (int j = 0; j < 4; ++j) Piece<TT>::unpack(kq[j], kf[j]);
#pragma unroll
      for (int g = 0; g < GM; ++g) {
        if (g < a.group) {
          float qf[N];
          Piece<TT>::unpack(*reinterpret_cast<const uint4*>(qp + (long long)g * a.d + i), qf);
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < N; ++e) acc[j][g] = fmaf(kf[j][e], qf[e], acc[j][g]);
        }
      }
    }
  } else {
    for (int i = l8; i < a.d; i += 8) {
      float kf[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) kf[j] = ld_elem<TT>(kp[j], i);
#pragma unroll
      for (int g = 0; g < GM; ++g) {
        if (g < a.group) {
          const float qf = ld_elem<TT>(qp + (long long)g * a.d, i);
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[j][g] = fmaf(kf[j], qf, acc[j][g]);
        }
      }
    }
  }
#pragma unroll
  for (int g = 0; g < GM; ++g) {
    if (g < a.group) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float v = acc[j][g];
#pragma unroll
        for (int o = 4; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (l8 == 0) s_logit[g][r0 + 32 * j] = v * a.scale;
      }
    }
  }
  __syncthreads();
  // a warp per head: 128 logits, four a lane
  for (int g = warp; g < a.group; g += 8) {
    float v[4], m = -INFINITY, s = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) { v[j] = lane + 32 * j < n_tok ? s_logit[g][lane + 32 * j] : -INFINITY; m = fmaxf(m, v[j]); }
#pragma unroll
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (lane + 32 * j < n_tok) s += expf(v[j] - finite_or_zero(m));
#pragma unroll
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0)
      a.stats[(stats_block(sq.seq_off[b], a.seq_base + b) + blockIdx.x / (unsigned)a.n_kv) * a.n_heads + kvh * a.group + g] = make_float2(m, s);
  }
  for (int i = threadIdx.x; i < a.group * A_TOK; i += 256) {
    const int g = i / A_TOK, r = i % A_TOK;
    if (r < n_tok) a.logits[((long long)kvh * a.group + g) * a.T_total + t0 + r] = s_logit[g][r];
  }
}

constexpr int A_HEADS = 16;
// (max, sum exp) of two disjoint sets
__device__ __forceinline__ float2 merge_stats(float2 p, float2 q) {
  const float m = fmaxf(p.x, q.x), mf = finite_or_zero(m);
  return make_float2(m, p.y * expf(p.x - mf) + q.y * expf(q.x - mf));
}
// (max, 1 / sum exp) over a sequence of nh <= A_TOK heads, from those of its blocks at `st`, to s_ms; as many threads a head as there are,
// added up in a fixed order.  By all threads of a CTA of A_TOK, which may use s_ms behind it.
__device__ __forceinline__ void merge_blocks(const float2* st, int n_blk, int n_heads, int nh, float2* s_part, float2* s_ms) {
  const int per = nh <= 16 ? 16 : nh <= 32 ? 32 : nh <= 64 ? 64 : 128, parts = A_TOK / per;      // heads side by side; threads a head
  const int hl = threadIdx.x & (per - 1), part = threadIdx.x / per;
  float2 ms = make_float2(-INFINITY, 0.f);
  for (int k = part; k < n_blk; k += 4 * parts) {      // four blocks in flight
    float2 p[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      p[j] = k + j * parts < n_blk && hl < nh ? st[(long long)(k + j * parts) * n_heads + hl] : make_float2(-INFINITY, 0.f);
    ms = merge_stats(ms, merge_stats(merge_stats(p[0], p[1]), merge_stats(p[2], p[3])));
  }
  s_part[threadIdx.x] = ms;
  __syncthreads();
  if (threadIdx.x < per) {
    for (int q = 1; q < parts; ++q) ms = merge_stats(ms, s_part[q * per + threadIdx.x]);
    s_ms[threadIdx.x] = make_float2(ms.x, ms.y > 0.f ? 1.f / ms.y : 0.f);
  }
  __syncthreads();
}

// The statistics of a sequence, a warp per head, over those of its first block: a lane takes every 32nd block, four in flight, then five exchanges.
constexpr int A_MW = 4;        // warps a CTA
__global__ void __launch_bounds__(A_MW * 32) attn_merge_kernel(const AttnDev a, const AttnSeqs sq) {
  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.y, h = blockIdx.x * A_MW + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const long long lo = sq.seq_off[b], hi = sq.seq_off[b + 1];
  if (hi == lo || h >= a.n_heads) return;
  const int n_blk = (int)((hi - lo + A_TOK - 1) / A_TOK);
  float2* st = a.stats + stats_block(lo, a.seq_base + b) * a.n_heads + h;
  float2 ms = make_float2(-INFINITY, 0.f);
  for (int k = lane; k < n_blk; k += 4 * 32) {
    float2 p[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) p[j] = k + j * 32 < n_blk ? st[(long long)(k + j * 32) * a.n_heads] : make_float2(-INFINITY, 0.f);
    ms = merge_stats(ms, merge_stats(merge_stats(p[0], p[1]), merge_stats(p[2], p[3])));
  }
#pragma unroll
  for (int o = 16; o; o >>= 1)
    ms = merge_stats(ms, make_float2(__shfl_xor_sync(0xffffffffu, ms.x, o), __shfl_xor_sync(0xffffffffu, ms.y, o)));
  if (lane == 0) st[0] = make_float2(ms.x, ms.y > 0.f ? 1.f / ms.y : 0.f);
}

// A CTA per 128 tokens, sixteen heads at a time: their logits of the thread's token are asked for, then (MERGED: read; else formed from the
// blocks', of all heads at once) each head's maximum and sum over the sequence, then the terms.  What bounds it is the latency of
// its two rounds of loads.
template <bool MERGED>
__global__ void __launch_bounds__(A_TOK) attn_average_kernel(const AttnDev a, const AttnSeqs sq) {
  __shared__ float2 s_part[A_TOK], s_ms[A_TOK];
  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.y;
  const long long lo = sq.seq_off[b], hi = sq.seq_off[b + 1], t0 = lo + (long long)blockIdx.x * A_TOK, t = t0 + threadIdx.x;
  if (t0 >= hi) return;
  const bool on = t < hi;
  const float2* st = a.stats + stats_block(lo, a.seq_base + b) * a.n_heads;
  const float* l = a.logits + t;
  float acc = 0.f;
  for (int h0 = 0; h0 < a.n_heads; h0 += A_HEADS) {
    const int nh = min(A_HEADS, a.n_heads - h0);
    float v[A_HEADS];
    float2 ms[A_HEADS];
#pragma unroll
    for (int i = 0; i < A_HEADS; ++i) {
      v[i] = on && i < nh ? l[(long long)(h0 + i) * a.T_total] : 0.f;
      if (MERGED && i < nh) ms[i] = st[h0 + i];
    }
    if (!MERGED && h0 % A_TOK == 0) merge_blocks(st + h0, (int)((hi - lo + A_TOK - 1) / A_TOK), a.n_heads, min(A_TOK, a.n_heads - h0), s_part, s_ms);
#pragma unroll
    for (int i = 0; i < A_HEADS; ++i) {
      const float2 p = MERGED ? ms[i] : s_ms[h0 % A_TOK + i];
      if (i < nh) acc += expf(v[i] - p.x) * p.y;
    }
  }
  if (on) a.out[t] = acc / (float)a.n_heads;
}

template <typename TT, bool VEC>
static cudaError_t launch_logits(const AttnDev& a, const AttnSeqs& sq, long long max_len, int nb, cudaStream_t s) {
  const dim3 grid((unsigned)((max_len + A_TOK - 1) / A_TOK * a.n_kv), (unsigned)nb), block(256);
  if (a.group == 1) return launch_pdl(attn_logits_kernel<TT, 1, VEC>, grid, block, 0, s, 1, a, sq);
  if (a.group <= 4) return launch_pdl(attn_logits_kernel<TT, 4, VEC>, grid, block, 0, s, 1, a, sq);
  if (a.group <= 8) return launch_pdl(attn_logits_kernel<TT, 8, VEC>, grid, block, 0, s, 1, a, sq);
  return launch_pdl(attn_logits_kernel<TT, 16, VEC>, grid, block, 0, s, 1, a, sq);
}

}  // namespace fmmoe

using namespace fmmoe;

extern "C" __attribute__((visibility("default"))) size_t fmmoe_attention_workspace_bytes(int64_t n_tokens, int32_t n_seq,
                                                                                         int32_t n_heads) {
  if (n_tokens < 0 || n_seq < 0 || n_heads < 1) return 0;
  return align_up((size_t)n_tokens * n_heads * 4, 256) + align_up((size_t)stats_block(n_tokens, n_seq) * n_heads * 8, 256) + 256;
}

extern "C" __attribute__((visibility("default"))) fmmoe_status fmmoe_attention_importance(
    fmmoe_handle* h, const void* q_last, const void* k, int32_t dtype, int32_t n_heads, int32_t n_kv_heads,
    int32_t head_dim, float scale, const int64_t* seq_off, int32_t n_seq, float* attn_out, void* workspace,
    size_t workspace_bytes, void* cuda_stream) {
  if (!h || !seq_off || n_seq < 0 || n_heads < 1 || n_kv_heads < 1 || head_dim < 1) return FMMOE_ERR_INVALID_ARG;
  if (dtype != FMMOE_F32 && dtype != FMMOE_BF16) return FMMOE_ERR_INVALID_ARG;
  if (n_heads % n_kv_heads) return FMMOE_ERR_INVALID_ARG;
  if (n_heads / n_kv_heads > A_MAX_GROUP) return FMMOE_ERR_UNSUPPORTED;
  if (n_seq && seq_off[0] != 0) return FMMOE_ERR_INVALID_ARG;
  for (int b = 0; b < n_seq; ++b)
    if (seq_off[b + 1] < seq_off[b]) return FMMOE_ERR_INVALID_ARG;
  const int64_t T = n_seq ? seq_off[n_seq] : 0;
  if (T == 0) return FMMOE_OK;
  if (!q_last || !k || !attn_out) return FMMOE_ERR_INVALID_ARG;
  const size_t need = fmmoe_attention_workspace_bytes(T, n_seq, n_heads) - 256;
  if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < need) return FMMOE_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  char* ws = static_cast<char*>(workspace);
  AttnDev a = {};
  a.q = q_last; a.k = k; a.n_heads = n_heads; a.n_kv = n_kv_heads; a.d = head_dim; a.group = n_heads / n_kv_heads;
  a.scale = scale; a.logits = reinterpret_cast<float*>(ws);
  a.stats = reinterpret_cast<float2*>(ws + align_up((size_t)T * n_heads * 4, 256));
  a.out = attn_out; a.T_total = T;
  // 16-byte pieces need rows and pointers that are multiples of 16 bytes; the library asks for neither here
  const bool vec = ((size_t)head_dim * (dtype == FMMOE_BF16 ? 2 : 4)) % 16 == 0 && (((uintptr_t)q_last | (uintptr_t)k) & 15) == 0;
  for (int b0 = 0; b0 < n_seq; b0 += A_MAXS) {
    const int nb = n_seq - b0 < A_MAXS ? n_seq - b0 : A_MAXS;
    AttnSeqs sq = {};
    sq.n_seq = nb;
    for (int i = 0; i <= nb; ++i) sq.seq_off[i] = seq_off[b0 + i];
    a.seq_base = b0;
    const long long n_tok = sq.seq_off[nb] - sq.seq_off[0];
    if (n_tok == 0) continue;
    long long max_len = 0;
    for (int i = 0; i < nb; ++i) max_len = sq.seq_off[i + 1] - sq.seq_off[i] > max_len ? sq.seq_off[i + 1] - sq.seq_off[i] : max_len;
    // The merge kernel is a launch more, but without it every average CTA goes over the statistics of the whole sequence.  Bounds in blocks x heads, without
    // / with it, us in a graph: 16 heads on 4 kv heads: 2,432 tokens (304) 6.3 / 6.8, eight such sequences 10.5 / 10.9, 8,192 (1,024) 8.2 / 8.0, 16,384 12.1 /
    // 10.7; 32 on 8: 686 tokens (192) 8.4 / 8.8, 2,432 (608) 10.1 / 9.9, 16,384 23.9 / 19.1; 64 on 4: 256 tokens (128) 14.0 / 14.1, 686 (384) 14.8 / 14.7, 2,432
    // 17.2 / 15.3.  A kv head per head has as many logits CTAs as average CTAs x heads: 16 heads, 686 tokens 5.5 / 5.9, 2,432 8.1 / 6.9, eight such 19.3 / 17.4.
    const long long blocks = (max_len + A_TOK - 1) / A_TOK;
    const bool merged = blocks * n_heads > 320 || (a.group == 1 && blocks > 8);
    {
      ProfScope ps(h, FMMOE_KERNEL_ATTN, s);
      if (dtype == FMMOE_BF16) FMMOE_CUDA_TRY((vec ? launch_logits<__nv_bfloat16, true> : launch_logits<__nv_bfloat16, false>)(a, sq, max_len, nb, s));
      else FMMOE_CUDA_TRY((vec ? launch_logits<float, true> : launch_logits<float, false>)(a, sq, max_len, nb, s));
      if (merged) FMMOE_CUDA_TRY(launch_pdl(attn_merge_kernel, dim3((unsigned)((n_heads + A_MW - 1) / A_MW), nb), dim3(A_MW * 32), 0, s, 1, a, sq));
      FMMOE_CUDA_TRY(launch_pdl(merged ? attn_average_kernel<true> : attn_average_kernel<false>, dim3((unsigned)((max_len + A_TOK - 1) / A_TOK), nb), dim3(A_TOK), 0, s, 1, a, sq));
    }
    FMMOE_CUDA_TRY(cudaGetLastError());
    h->launches += merged ? 3 : 2;
  }
  return FMMOE_OK;
}
