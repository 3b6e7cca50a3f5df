// Routing-aware sliding-window pruning of vision tokens (Section 3.2).
//   window_score_kernel: per window, its member tokens (a scan of the mask up to them), routing similarity
//                        S (Eq. 8 or Eq. 9-10) and the attention sum (Eq. 11); one warp per window, fp64
//   select_kernel      : per sequence, ranks of the vision tokens, A_bar (Eq. 12), C (Eq. 13) rounded once to
//                        fp32, merge set = m highest C (Eq. 15), drop set = d smallest A_bar among the rest
//                        (both by a search for the bounding (score, window) key), then the stable compaction
//                        map (scan of keep flags) and the list of merged rows
//   compact_kernel     : copies kept rows (a warp per row); a merged window becomes mean(rows) rescaled to the
//                        largest member norm (Eq. 16-18) at its first token's position (a CTA per window)
// The (score, window index) keys are unique, so the keep-set does not depend
// on thread order; ties go to the lower window index.
#include <cuda_bf16.h>
#include <math.h>
#include <pthread.h>

#include "internal.h"
#include "ptx.cuh"

namespace fmmoe {

constexpr int MAXS = FMMOE_MAX_SEQS_PER_LAUNCH;
constexpr int MAXW = FMMOE_MAX_WINDOW;

struct PruneDev {
  const float* probs; const float* attn; const void* x; const uint8_t* is_visual;
  int E, H, W, sim_mode, merge_mode, dtype;
  double alpha;
  // workspace
  int2* merges;        // [windows] of each sequence, the first m entries: (output row, rank of the first member)
  int32_t* vis_list;   // [T] token index of the v-th vision token of sequence b at seq_off[b]+v
  double* sim;         // [windows]
  double* asum;        // [windows]
  // outputs
  void* x_out; uint8_t* is_visual_out; int32_t* keep_idx; uint8_t* kind;
  int32_t* keep_idx_ws; uint8_t* kind_ws;   // always-present copies in the workspace
  int32_t* pos;        // not NULL: the inverse map instead, [T] output row of a copied token, -1 for others
  int late;            // compact_kernel writes is_visual_out, keep_idx and kind (NULL for select_kernel): one of them lies
                       // over is_visual, which other threads and CTAs of select_kernel may still have to read
  int* status;
};

// ------------------------------------------------------------------ window scores
// Window i of a sequence from its members' routing rows.  The W(W+1)/2 dot products (lower triangle, q = i(i+1)/2 + j)
// are summed over the lanes so that lane q ends up with product q (31 shuffles for up to 32 products instead of five
// each), and every lane then forms the cosine of its own pair: one division and two roots deep whatever W is.
template <int W>
__device__ __forceinline__ void score_window(const PruneDev& a, const int32_t* members, int lane, double* sim_out,
                                             double* asum_out) {
  constexpr int NP = W * (W + 1) / 2;
  constexpr int NL = NP > 32 ? 32 : NP;                                   // products held one per lane
  constexpr int P2 = NL > 16 ? 32 : NL > 8 ? 16 : NL > 4 ? 8 : NL > 2 ? 4 : 2;
  double dots[NP > P2 ? NP : P2];
#pragma unroll
  for (int i = 0; i < (NP > P2 ? NP : P2); ++i) dots[i] = 0.0;
  const float* rows[W];
#pragma unroll
  for (int i = 0; i < W; ++i) rows[i] = a.probs + (long long)members[i] * a.E;
#pragma unroll 2
  for (int e = lane; e < a.E; e += 32) {
    double v[W];
#pragma unroll
    for (int i = 0; i < W; ++i) v[i] = (double)rows[i][e];
    int q = 0;
#pragma unroll
    for (int i = 0; i < W; ++i)
#pragma unroll
      for (int j = 0; j <= i; ++j) { dots[q] = fma(v[i], v[j], dots[q]); ++q; }
  }
  double asum = 0.0;
  if (a.attn) {
#pragma unroll
    for (int i = 0; i < W; ++i) asum += (double)a.attn[members[i]];
  }
#pragma unroll
  for (int i = 32; i < NP; ++i)                                           // W = 8: the last four, summed on every lane
#pragma unroll
    for (int o = 16; o; o >>= 1) dots[i] += __shfl_xor_sync(0xffffffffu, dots[i], o);
#pragma unroll
  for (int o = P2 / 2; o; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const double send = up ? dots[i] : dots[i + o], keep = up ? dots[i + o] : dots[i];
      dots[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  double mine = dots[0];
#pragma unroll
  for (int o = P2; o < 32; o <<= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  auto dot = [&](int q) {              // product q, on every lane
    double v = __shfl_sync(0xffffffffu, mine, q & 31);
#pragma unroll
    for (int k = 32; k < NP; ++k)
      if (q == k) v = dots[k];
    return v;
  };
  auto sum_lanes = [&](double v) {
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  double s = 0.0;
  if (a.sim_mode == 0) {
#pragma unroll
    for (int q0 = 0; q0 < NP; q0 += 32) {
      const int q = q0 + lane;
      int i = 0;
      while ((i + 1) * (i + 2) / 2 <= q) ++i;                             // row of product q
      const int j = q - i * (i + 1) / 2;
      const bool pair = q < NP && j < i;
      const double nn = sqrt(dot(min(i, W - 1) * (min(i, W - 1) + 3) / 2)) * sqrt(dot(min(j, W - 1) * (min(j, W - 1) + 3) / 2));
      const double d = dot(min(q, NP - 1));
      if (pair) s += d / nn;
    }
    s = sum_lanes(s) / (double)(W * (W - 1) / 2);
  } else {
    // mean row rbar = sum(rows)/W:  rows_i . rbar = sum_j D(i,j)/W ;  rbar . rbar = sum_ij D(i,j)/W^2
    const int i = min(lane, W - 1);
    double t = 0.0;
#pragma unroll
    for (int j = 0; j < W; ++j) t += dot(j <= i ? i * (i + 1) / 2 + j : j * (j + 1) / 2 + i);
    const double rr = sum_lanes(lane < W ? t : 0.0) / (double)(W * W);
    const double nn = sqrt(dot(i * (i + 3) / 2)) * sqrt(rr);
    s = sum_lanes(lane < W ? t / (double)W / nn : 0.0) / (double)W;
  }
  if (lane == 0) { *sim_out = s; *asum_out = asum; }
}

// A CTA scores eight windows of one sequence.  It finds their member tokens itself by counting the mask up to them
// (4,096 tokens a round, from L2), which costs less than a kernel of its own in front of this one.  What bounds it is
// the latency of that count, of one round of row loads and of the fp64 tail: 9.6 us for 665
// windows of 5 x 128 experts, 12.8 us for 6,144 windows of 3 x 64 in eight sequences (the rank kernel and a warp that
// formed all cosines on every lane took 6.2 + 10.5 and 5.1 + 11.3 us).  A kernel per W: registers go with W squared.
// MINB, the CTAs an SM that are asked for: six up to W = 3 (40 registers, no spills; 768 CTAs of eight sequences of 2,304 tokens are one wave, the
// stage 33.6 -> 31.8 us), else one, for which the compiler takes 64, 82, 109, 128 and 153 registers from W = 4 on, or zero: nothing is asked for
// and it takes 64 for W = 5 and 128 for W = 8, with which four and two CTAs fit an SM instead of two and one.
// score_kernel says when.
template <int W, int MINB>
__global__ void __launch_bounds__(256, MINB) window_score_kernel(const PruneDev a, const PruneSeqs sq) {
  __shared__ int s_mem[SC_WIN * W];
  __shared__ int s_cnt[128];
  __shared__ int s_total;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.y;
  const int n_f = sq.win_off[b + 1] - sq.win_off[b];
  const int i0 = blockIdx.x * SC_WIN;
  pdl_launch_dependents();
  pdl_wait();
  if (i0 >= n_f) return;
  const long long lo = sq.seq_off[b], hi = sq.seq_off[b + 1];
  const int r0 = i0 * W, r1 = min(i0 + SC_WIN, n_f) * W;    // ranks of the vision tokens this CTA needs
  // entries that a mask with fewer set bytes than the host's count leaves open hold a token of the sequence
  if (tid < SC_WIN * W) s_mem[tid] = (int)lo;
  int running = 0;
  for (long long t0 = lo; t0 < hi && running < r1; t0 += 4096) {
    uint32_t bits = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const long long t = t0 + j * 256 + tid;
      if (t < hi && a.is_visual[t] != 0) bits |= 1u << j;
    }
    uint32_t bal[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) bal[j] = __ballot_sync(0xffffffffu, (bits >> j) & 1u);
    uint32_t own = 0;                                  // lane j of a warp keeps ballot j's count
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (lane == j) own = __popc(bal[j]);
    if (lane < 16) s_cnt[lane * 8 + warp] = (int)own;
    __syncthreads();
    if (warp == 0) {
      int c[4], sum = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) { c[k] = s_cnt[lane * 4 + k]; sum += c[k]; }
      int incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int n = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += n;
      }
      int at = incl - sum;
#pragma unroll
      for (int k = 0; k < 4; ++k) { s_cnt[lane * 4 + k] = at; at += c[k]; }
      if (lane == 31) s_total = incl;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int rank = running + s_cnt[j * 8 + warp] + __popc(bal[j] & ((1u << lane) - 1u));
      if (((bits >> j) & 1u) && rank >= r0 && rank < r1) s_mem[rank - r0] = (int)(t0 + j * 256 + tid);
    }
    running += s_total;
    __syncthreads();
  }
  const int i = i0 + warp;
  if (i >= n_f) return;
  score_window<W>(a, s_mem + warp * W, lane, a.sim + sq.win_off[b] + i, a.asum + sq.win_off[b] + i);
}

typedef void (*ScoreKernel)(const PruneDev, const PruneSeqs);
static const ScoreKernel kScore[MAXW - 1] = {window_score_kernel<2, 6>, window_score_kernel<3, 6>, window_score_kernel<4, 1>,
                                             window_score_kernel<5, 0>, window_score_kernel<6, 1>, window_score_kernel<7, 1>,
                                             window_score_kernel<8, 0>};
static const ScoreKernel kScoreFew[2] = {window_score_kernel<5, 1>, window_score_kernel<8, 1>};
// More registers a thread hide more of a window's latency as long as the CTAs still fit the chip at once; beside a layer's GEMMs they get one SM or a few and
// what the GEMMs leave.  A stage alone, 64 experts, fewer / more registers, us: W = 5: eight sequences of 1,100 tokens (224 CTAs) 21.0 / 18.7, one of 8,000 (200)
// 41.0 / 39.5, sixteen of 950 (384) 21.2 / 21.7, eight of 2,304 (464) 32.1 / 35.0, 64 of 950 (1,536) 64.1 / 72.1; W = 8: 1,100 (144) 20.7 / 19.3, 8,000 (125) 34.2 / 33.4, sixteen of 950
// (240) 20.6 / 23.7, 2,304 (288) 32.9 / 37.7.  Beside the GEMMs, W = 5, 3,400 tokens: the layer 274 / 287.
static ScoreKernel score_kernel(int W, int64_t ctas, int sm_count, bool alone) {
  if (alone && W == 5 && ctas <= 2 * sm_count) return kScoreFew[0];
  if (alone && W == 8 && ctas <= sm_count) return kScoreFew[1];
  return kScore[W - 2];
}

// ------------------------------------------------------------------ select + compaction map
// Order-preserving map float -> uint32 (-0 is folded onto +0 so that equal values tie).
__device__ __forceinline__ uint32_t ordered_bits(float f) {
  if (f == 0.f) f = 0.f;
  const uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Block-wide count of n keys below a bound: the thread's own key (n <= THREADS), or the keys in shared memory.  Every
// thread gets the result; `slot` alternates between two rows of s_w so that one barrier a call is enough.
template <int THREADS> struct KeyCount {
  const unsigned long long* keys; unsigned long long own; int n; bool in_regs; int (*s_w)[32]; int slot;
  __device__ __forceinline__ int below(unsigned long long bound) {
    if (in_regs) return __syncthreads_count(own < bound);
    int c = 0;
    for (int i = threadIdx.x; i < n; i += THREADS) c += keys[i] < bound;
    c = __reduce_add_sync(0xffffffffu, c);
    if ((threadIdx.x & 31) == 0) s_w[slot][threadIdx.x >> 5] = c;
    __syncthreads();
    const int v = (threadIdx.x & 31) < THREADS / 32 ? s_w[slot][threadIdx.x & 31] : 0;
    slot ^= 1;
    return __reduce_add_sync(0xffffffffu, v);
  }
};

// A bound that exactly k of the (unique) keys lie below, 1 <= k <= number of keys that are not ~0.  Built bit by bit
// from the highest bit in which the keys' upper halves differ (`hi_and`, `hi_or`: their conjunction and disjunction);
// one barrier a step, and it ends as soon as a candidate has k keys below it (a dozen steps past the common prefix
// for distinct scores), where sorting 1,024 keys takes 55 steps, half of them with two barriers.
template <int THREADS>
__device__ __forceinline__ unsigned long long bound_of_k_smallest(KeyCount<THREADS>& kc, int k, uint32_t hi_and, uint32_t hi_or) {
  const uint32_t diff = hi_and ^ hi_or;
  const int top = diff ? 63 - __clz((int)diff) : 31;
  unsigned long long t = top == 63 ? 0ull : ((unsigned long long)hi_and << 32) & ~((2ull << top) - 1ull);
  for (int bit = top; bit >= 0; --bit) {
    const unsigned long long mid = t | (1ull << bit);
    const int c = kc.below(mid);
    if (c == k) return mid;
    if (c < k) t = mid;
  }
  return t + 1;     // t is the k-th smallest key itself
}

// Exclusive scan of one int per thread over the CTA; *total gets the sum.  s_w: 32 ints of shared memory.
template <int THREADS>
__device__ __forceinline__ int block_scan(int v, int* s_w, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += n;
  }
  if (lane == 31) s_w[warp] = incl;
  __syncthreads();
  int c = lane < THREADS / 32 ? s_w[lane] : 0;      // every warp scans the warp sums for itself
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int n = __shfl_up_sync(0xffffffffu, c, o);
    if (lane >= o) c += n;
  }
  *total = __shfl_sync(0xffffffffu, c, 31);
  const int before = __shfl_sync(0xffffffffu, c, warp ? warp - 1 : 0);
  return (warp ? before : 0) + incl - v;
}

// A selection CTA of 1,024 threads has all registers of an SM.  One of 256 has shorter barriers and, with 80 registers a thread (no spills; with the
// 64 that the compiler takes by itself it spills), fits beside a CTA of the bf16 small-M expert GEMMs, which leaves 20,480; beside those of the FP8
// weight stream, which leave 7,168, nothing of selection does.  That many threads do for sequences of at most 1,024 tokens (their mask stays in registers, four a
// thread) with a window a thread: 44 windows of 224 tokens 9.5 -> 7.1 us (before the rolled loops below).
constexpr int SEL_THREADS = 1024, SEL_SMALL = 256;
constexpr int64_t SEL_SMALL_TOKENS = 1024;
constexpr int64_t SEL_MAX_WINDOWS = 16384;    // of a sequence: nine bytes of shared memory each

// One CTA per sequence.  Ranks of the vision tokens, Eq. 12-13 (one rounding to fp32), then the merge set (Eq. 15)
// and the drop set as the keys below a bound.  A chain of barriers and of a few rounds of loads: 14.1 us
// for eight sequences of 768 windows with attention, 16.5 us for one of 665 and 3,584 tokens (24.5 and 26 us with two
// in-CTA sorts and ranks from memory).
template <int THREADS>      // windows whose keys stay in registers, one per thread: up to THREADS
__global__ void __launch_bounds__(THREADS, THREADS == SEL_SMALL ? 3 : 1) select_kernel(const PruneDev a, const PruneSeqs sq) {
  extern __shared__ unsigned long long s_keys[];   // [n_f] keys (more than THREADS windows), then [n_f] action bytes
  __shared__ double s_red[32];
  __shared__ int s_scan[2][32];
  __shared__ int s_w[2][32];
  __shared__ uint32_t s_hi[2][2][32];
  __shared__ int s_merged;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_launch_dependents();
  const int n_f = sq.n_vis[b] / a.W;
  const int w0 = sq.win_off[b];
  const int m = sq.m[b], d = sq.d[b];
  const bool have_attn = a.attn != nullptr;
  const bool in_regs = n_f <= THREADS;
  uint8_t* s_action = reinterpret_cast<uint8_t*>(s_keys + (in_regs ? 0 : n_f));   // [n_f]
  const long long lo = sq.seq_off[b], hi = sq.seq_off[b + 1];
  const int per = (int)((hi - lo + THREADS - 1) / THREADS);      // every thread owns a run of consecutive tokens
  const long long t_begin = lo + (long long)tid * per;
  // The mask of the run's first tokens stays in a register, and later what is emitted for them, two bits a token.  The loops over
  // them are not unrolled and the window of the next vision token is carried along: a thread owns one token to a few, and eight copies
  // of a body with a division in it cost more than they saved.  One sequence of 256 tokens 7.0 -> 5.6 us, a pruned fp32 layer of
  // 256 tokens 39.8 -> 37.9 us, the stage of eight sequences of 2,400 tokens 45.7 -> 45.1 us.
  constexpr int CACHE = 8;
  const int n_own = (int)min((long long)per, max(hi - t_begin, 0ll)), n_cached = min(n_own, CACHE);
  if (tid == 0) s_merged = 0;
  pdl_wait();
  uint32_t vis = 0;
#pragma unroll
  for (int i = 0; i < CACHE; ++i)
    if (i < n_own && a.is_visual[t_begin + i] != 0) vis |= 1u << i;
  double my_s = 0.0, my_a = 0.0;                       // in_regs: this thread's window
  if (in_regs && tid < n_f) { my_s = a.sim[w0 + tid]; if (have_attn) my_a = a.asum[w0 + tid]; }
  for (int i = tid; i < m; i += THREADS) a.merges[w0 + i] = make_int2(-1, 0);
  for (int i = tid; i < n_f; i += THREADS) s_action[i] = 0;
  if (a.pos)
    for (long long t = lo + tid; t < hi; t += THREADS) a.pos[t] = -1;     // several barriers before the first row is placed

  // vision ranks
  int n_mine = __popc(vis);
  for (int i = CACHE; i < n_own; ++i)
    if (a.is_visual[t_begin + i] != 0) ++n_mine;
  int found;
  const int rank0 = block_scan<THREADS>(n_mine, s_scan[0], &found);
  {
    int r = rank0;
    for (uint32_t left = vis; left; left &= left - 1) a.vis_list[lo + r++] = (int32_t)(t_begin + __ffs((int)left) - 1);
    for (int i = CACHE; i < n_own; ++i)
      if (a.is_visual[t_begin + i] != 0) a.vis_list[lo + r++] = (int32_t)(t_begin + i);
  }
  // A mask with fewer set bytes than the host's count leaves the tail of this sequence's list unwritten;
  // the merge kernel indexes x with these entries, so they must hold a token of the
  // sequence whatever the mask says (the mismatch itself is reported through the status word).
  for (int i = found + tid; i < sq.n_vis[b]; i += THREADS) a.vis_list[lo + i] = (int32_t)lo;
  if (tid == 0 && found != sq.n_vis[b]) atomicCAS(a.status, 0, DEV_INTERNAL);

  // Eq. 12: divide by the largest window sum (0 if all sums are 0)
  double amax = 0.0;
  if (have_attn) {
    if (in_regs) amax = fmax(amax, my_a);
    else for (int i = tid; i < n_f; i += THREADS) amax = fmax(amax, a.asum[w0 + i]);
#pragma unroll
    for (int o = 16; o; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if (lane == 0) s_red[warp] = amax;
    __syncthreads();
    amax = lane < THREADS / 32 ? s_red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o; o >>= 1) amax = fmax(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  }
  // key of the redundancy ranking: (C descending, window ascending); Eq. 13 in fp64 without
  // contraction, then ONE rounding to fp32
  auto c_key = [&](int i, double S, double A) -> unsigned long long {
    float c32;
    if (have_attn) {
      const double ab = amax > 0.0 ? A / amax : 0.0;
      c32 = (float)__dsub_rn(__dmul_rn(a.alpha, S), __dmul_rn(__dsub_rn(1.0, a.alpha), ab));
    } else {
      c32 = (float)S;
    }
    return ((unsigned long long)(~ordered_bits(c32)) << 32) | (unsigned)i;
  };
  // key of the drop ranking among the windows that were not merged: (A_bar ascending, window ascending)
  auto a_key = [&](int i, double A) -> unsigned long long {
    const float a32 = (float)(amax > 0.0 ? A / amax : 0.0);
    return ((unsigned long long)ordered_bits(a32) << 32) | (unsigned)i;
  };
  if (m + d > 0) {
    KeyCount<THREADS> kc = {s_keys, ~0ull, n_f, in_regs, s_w, 0};
    for (int pass = 0; pass < 2; ++pass) {             // 0: by C, 1: by A_bar among the rest
      if (pass == 1 && (!have_attn || d == 0)) break;
      uint32_t h_and = 0xffffffffu, h_or = 0;
      for (int i = tid; i < n_f; i += THREADS) {
        unsigned long long k = ~0ull;
        if (pass == 0) k = in_regs ? c_key(i, my_s, my_a) : c_key(i, a.sim[w0 + i], have_attn ? a.asum[w0 + i] : 0.0);
        else if (s_action[i] == 0) k = a_key(i, in_regs ? my_a : a.asum[w0 + i]);
        if (in_regs) kc.own = k; else s_keys[i] = k;
        if (k != ~0ull) { h_and &= (uint32_t)(k >> 32); h_or |= (uint32_t)(k >> 32); }
      }
      h_and = __reduce_and_sync(0xffffffffu, h_and);
      h_or = __reduce_or_sync(0xffffffffu, h_or);
      if (lane == 0) { s_hi[pass][0][warp] = h_and; s_hi[pass][1][warp] = h_or; }
      __syncthreads();                                 // the keys and the halves' bits are there
      h_and = __reduce_and_sync(0xffffffffu, lane < THREADS / 32 ? s_hi[pass][0][lane] : 0xffffffffu);
      h_or = __reduce_or_sync(0xffffffffu, lane < THREADS / 32 ? s_hi[pass][1][lane] : 0u);
      unsigned long long first = 0, second = 0;
      if (pass == 0) {
        if (m > 0) first = bound_of_k_smallest(kc, m, h_and, h_or);
        if (!have_attn && d > 0) second = bound_of_k_smallest(kc, m + d, h_and, h_or);
      } else {
        second = bound_of_k_smallest(kc, d, h_and, h_or);
      }
      for (int i = tid; i < n_f; i += THREADS) {
        const unsigned long long k = in_regs ? kc.own : s_keys[i];
        if (k < first) s_action[i] = 1;
        else if (k < second) s_action[i] = 2;
      }
      if (in_regs) kc.own = ~0ull;
      __syncthreads();
    }
  }

  // stable compaction map over the sequence's tokens
  int win, place;                      // window and place in it of the next vision token
  auto at_rank = [&](int v) { win = v / a.W; place = v - win * a.W; };
  auto next_kind = [&](bool v) -> int {      // kind of the row emitted for the next token, -1 = nothing emitted
    if (!v) return 0;
    const int act = win < n_f ? s_action[win] : 0, first = place == 0;
    if (++place == a.W) { place = 0; ++win; }
    return act == 0 ? 1 : act == 1 && first ? 2 : -1;
  };
  at_rank(rank0);
  uint32_t kinds = 0;                  // of the first tokens, plus one, two bits each
  int cnt = 0;
#pragma unroll 1
  for (int i = 0; i < n_cached; ++i) {
    const int k = next_kind((vis >> i) & 1u);
    kinds |= (uint32_t)(k + 1) << (2 * i);
    cnt += k >= 0;
  }
#pragma unroll 1
  for (int i = CACHE; i < n_own; ++i) cnt += next_kind(a.is_visual[t_begin + i] != 0) >= 0;
  int total;
  long long pos = sq.out_off[b] + block_scan<THREADS>(cnt, s_scan[1], &total);
  auto emit = [&](long long t, int kd, int rank) {
    if (pos < sq.out_off[b + 1]) {
      if (a.pos) {
        if (kd != 2) a.pos[t] = (int32_t)pos;
      } else {
        a.keep_idx_ws[pos] = (int32_t)t;
        a.kind_ws[pos] = (uint8_t)kd;
      }
      if (a.keep_idx) a.keep_idx[pos] = (int32_t)t;
      if (a.kind) a.kind[pos] = (uint8_t)kd;
      if (a.is_visual_out) a.is_visual_out[pos] = kd != 0;
      if (kd == 2) {
        const int i = atomicAdd(&s_merged, 1);         // any order: each entry writes a row of its own
        if (i < m) a.merges[w0 + i] = make_int2((int)pos, rank);
      }
    }
    ++pos;
  };
  int r = rank0;
#pragma unroll 1
  for (int i = 0; i < n_own; ++i) {
    bool v;
    int kd;
    if (i < CACHE) {
      v = (vis >> i) & 1u;
      kd = (int)((kinds >> (2 * i)) & 3u) - 1;
    } else {
      if (i == CACHE) at_rank(r);
      v = a.is_visual[t_begin + i] != 0;
      kd = next_kind(v);
    }
    if (kd >= 0) emit(t_begin + i, kd, r);
    r += v;
  }
  if (tid == 0 && total != (int)(sq.out_off[b + 1] - sq.out_off[b])) atomicCAS(a.status, 0, DEV_INTERNAL);
}

// ------------------------------------------------------------------ gather / merge rows
template <typename T> struct Row8;   // 8 elements (bf16) or 4 elements (fp32) per 16 bytes
template <> struct Row8<__nv_bfloat16> {
  static constexpr int N = 8;
  static __device__ __forceinline__ void unpack(const uint4 u, float* f) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[i]));
      f[2 * i] = v.x; f[2 * i + 1] = v.y;
    }
  }
  static __device__ __forceinline__ void store(__nv_bfloat16* p, const float* f) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
      w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
  }
};
template <> struct Row8<float> {
  static constexpr int N = 4;
  static __device__ __forceinline__ void unpack(const uint4 u, float* f) {
    f[0] = __uint_as_float(u.x); f[1] = __uint_as_float(u.y); f[2] = __uint_as_float(u.z); f[3] = __uint_as_float(u.w);
  }
  static __device__ __forceinline__ void store(float* p, const float* f) {
    *reinterpret_cast<float4*>(p) = make_float4(f[0], f[1], f[2], f[3]);
  }
};

// The first CTAs form one merged window each (their dependent steps are the longest), the others copy CP_ROWS rows of
// the output, a warp per row with all its loads in flight; rows of merged windows are skipped there.
// Bound by bytes at batch, by two rounds of loads below: 14.3 us for 5,517 rows of 4 KB with 921 merged windows (45 MB
// moved), 8.3 us for 2,753 rows with 62; 22.3 and 13.3 us when a CTA formed the merged rows among its four rows.
constexpr int CP_ROWS = 8;

template <typename T>
__global__ void __launch_bounds__(256, 4) compact_kernel(const PruneDev a, const PruneSeqs sq, int n_merges, long long row_base,
                                                      long long n_rows) {
  constexpr int N = Row8<T>::N;
  __shared__ float s_red[8][MAXW + 1];
  pdl_launch_dependents();
  pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const T* X = static_cast<const T*>(a.x);
  const int vec = a.H / N;                       // 16-byte pieces per row
  if ((int)blockIdx.x >= n_merges) {
    const long long rel = (long long)((int)blockIdx.x - n_merges) * CP_ROWS + warp;
    if (rel >= n_rows) return;
    const long long row = row_base + rel;
    const long long t0 = a.keep_idx_ws[row];
    const uint8_t kd = a.kind_ws[row];
    if (a.late && lane == 0) {
      if (a.keep_idx) a.keep_idx[row] = (int32_t)t0;
      if (a.kind) a.kind[row] = kd;
      if (a.is_visual_out) a.is_visual_out[row] = kd != 0;
    }
    if (kd == 2) return;
    int b = 0;
    while (b + 1 < sq.n_seq && row >= sq.out_off[b + 1]) ++b;
    uint4* dst = reinterpret_cast<uint4*>(static_cast<T*>(a.x_out) + row * a.H);
    if (t0 < sq.seq_off[b] || t0 >= sq.seq_off[b + 1]) {
      // a slot the selection pass did not fill: only possible when the mask contradicts the host's vision
      // count (reported through the status word).  Never index x with it.
      for (int i = lane; i < vec; i += 32) dst[i] = make_uint4(0u, 0u, 0u, 0u);
      return;
    }
    const uint4* src = reinterpret_cast<const uint4*>(X + t0 * a.H);
    for (int i0 = 0; i0 < vec; i0 += 256) {
      uint4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) { const int i = i0 + u * 32 + lane; if (i < vec) v[u] = src[i]; }
#pragma unroll
      for (int u = 0; u < 8; ++u) { const int i = i0 + u * 32 + lane; if (i < vec) dst[i] = v[u]; }
    }
    return;
  }
  // ---- a merged window
  int b = 0, k0 = (int)blockIdx.x;
  while (b + 1 < sq.n_seq && k0 >= sq.m[b]) { k0 -= sq.m[b]; ++b; }
  const int2 e = a.merges[sq.win_off[b] + k0];
  if (e.x < sq.out_off[b] || e.x >= sq.out_off[b + 1]) return;   // open entry: inconsistent mask / count (status word set)
  const int v0 = e.y < 0 || e.y + a.W > sq.n_vis[b] ? 0 : e.y;   // same: stay inside the list
  T* O = static_cast<T*>(a.x_out) + (long long)e.x * a.H;
  const long long s_lo = sq.seq_off[b], s_hi = sq.seq_off[b + 1];
  int mem[MAXW];
#pragma unroll
  for (int k = 0; k < MAXW; ++k) {
    mem[k] = k < a.W ? a.vis_list[s_lo + v0 + k] : (int)s_lo;
    if (mem[k] < s_lo || mem[k] >= s_hi) mem[k] = (int)s_lo;
  }
  const float invW = 1.f / (float)a.W;
  float part[MAXW + 1];
#pragma unroll
  for (int k = 0; k <= MAXW; ++k) part[k] = 0.f;
  // The CTA's first 256 pieces (every row of up to 4 KB) stay in registers between the norm pass and the store; longer
  // rows are read again.  Squared norms of the members and of the mean:
  float mean0[N];
  for (int i = tid; i < vec; i += 256) {
    float mean[N];
#pragma unroll
    for (int j = 0; j < N; ++j) mean[j] = 0.f;
#pragma unroll
    for (int kq = 0; kq < MAXW; kq += 4) {               // four member rows in flight
      uint4 raw[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (kq + k < a.W) raw[k] = *reinterpret_cast<const uint4*>(X + (long long)mem[kq + k] * a.H + i * N);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (kq + k < a.W) {
          float f[N];
          Row8<T>::unpack(raw[k], f);
#pragma unroll
          for (int j = 0; j < N; ++j) { part[kq + k] = fmaf(f[j], f[j], part[kq + k]); mean[j] += f[j]; }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const float mv = mean[j] * invW;
      part[MAXW] = fmaf(mv, mv, part[MAXW]);
      if (i < 256) mean0[j] = mean[j];
    }
  }
#pragma unroll
  for (int k = 0; k <= MAXW; ++k) {
    if (k < a.W || k == MAXW) {
#pragma unroll
      for (int o = 16; o; o >>= 1) part[k] += __shfl_xor_sync(0xffffffffu, part[k], o);
      if (lane == 0) s_red[warp][k] = part[k];
    }
  }
  __syncthreads();
  // every thread sums the eight warps' shares in the same order
  float nmax = 0.f, nb = 0.f;
#pragma unroll
  for (int k = 0; k <= MAXW; ++k) {
    if (k < a.W || k == MAXW) {
      float tot = 0.f;
#pragma unroll
      for (int ww = 0; ww < 8; ++ww) tot += s_red[ww][k];
      if (k < MAXW) nmax = fmaxf(nmax, sqrtf(tot)); else nb = sqrtf(tot);
    }
  }
  const float scale = (a.merge_mode == 1 ? 1.f : (nb > 0.f ? nmax / nb : 0.f)) * invW;   // Eq. 18
  for (int i = tid; i < vec; i += 256) {
    float mean[N];
    if (i < 256) {
#pragma unroll
      for (int j = 0; j < N; ++j) mean[j] = mean0[j];
    } else {
#pragma unroll
      for (int j = 0; j < N; ++j) mean[j] = 0.f;
#pragma unroll
      for (int k = 0; k < MAXW; ++k) {
        if (k < a.W) {
          float f[N];
          Row8<T>::unpack(*reinterpret_cast<const uint4*>(X + (long long)mem[k] * a.H + i * N), f);
#pragma unroll
          for (int j = 0; j < N; ++j) mean[j] += f[j];
        }
      }
    }
#pragma unroll
    for (int j = 0; j < N; ++j) mean[j] *= scale;
    Row8<T>::store(O + i * N, mean);
  }
}

static int64_t counts_for(int64_t n_vis, int64_t n_retain, const fmmoe_prune_params* p, int64_t* m_out, int64_t* d_out) {
  const int64_t W = p->window;
  const int64_t eps = n_vis - n_retain;
  const int64_t n_f = n_vis / W;
  int64_t m = 0, d = 0;
  if (!(n_retain >= n_vis || eps <= W)) {
    if (p->merge_mode != 2) {
      m = (int64_t)floor((double)n_retain * p->gamma + 1e-9);
      if (m > eps / (W - 1)) m = eps / (W - 1);
      if (m > n_f) m = n_f;
      if (m < 0) m = 0;
    }
    const int64_t u = eps - m * (W - 1);
    d = u / W;
    if (d > n_f - m) d = n_f - m;
  }
  if (m_out) *m_out = m;
  if (d_out) *d_out = d;
  return n_vis - m * (W - 1) - d * W;
}

bool prune_outputs_over_mask(const uint8_t* is_visual, int64_t T, int64_t T_out, const uint8_t* is_visual_out,
                             const int32_t* keep_idx, const uint8_t* kind) {
  const uintptr_t m = (uintptr_t)is_visual;
  auto over = [&](const void* p, size_t elem) {
    return p && (uintptr_t)p < m + (uintptr_t)T && m < (uintptr_t)p + (uintptr_t)T_out * elem;
  };
  return over(is_visual_out, 1) || over(keep_idx, 4) || over(kind, 1);
}

}  // namespace fmmoe

using namespace fmmoe;

static bool prune_params_ok(const fmmoe_prune_params* p) {
  return p && p->window >= 2 && p->window <= FMMOE_MAX_WINDOW && p->sim_mode >= 0 && p->sim_mode <= 1 &&
         p->merge_mode >= 0 && p->merge_mode <= 2 && p->alpha >= 0.0 && p->alpha <= 1.0 && p->gamma >= 0.0;
}

extern "C" __attribute__((visibility("default"))) int64_t fmmoe_prune_kept_count(int64_t n_vis, int64_t n_retain, const fmmoe_prune_params* p,
                                          int64_t* n_merge, int64_t* n_drop) {
  if (!prune_params_ok(p) || n_vis < 0 || n_retain < 0) return -1;
  return counts_for(n_vis, n_retain, p, n_merge, n_drop);
}

extern "C" __attribute__((visibility("default"))) int64_t fmmoe_prune_output_rows(const fmmoe_prune_params* p, const int64_t* seq_off,
                                          const int64_t* n_vis, const int64_t* n_retain, int32_t n_seq) {
  if (!prune_params_ok(p) || n_seq < 0 || (n_seq && (!seq_off || !n_vis || !n_retain))) return INT64_MIN;
  int64_t rows = 0;
  for (int32_t b = 0; b < n_seq; ++b) {
    if (n_vis[b] < 0 || n_retain[b] < 0) return INT64_MIN;
    rows += seq_off[b + 1] - seq_off[b] - n_vis[b] + counts_for(n_vis[b], n_retain[b], p, nullptr, nullptr);
  }
  return rows;
}

namespace {
struct PruneWs { size_t merges, vis_list, sim, asum, keep_idx, kind, total; };
PruneWs plan_prune(int64_t T) {
  PruneWs w; size_t o = 0;
  const size_t nw = (size_t)T / 2 + 1;
  w.merges = o; o = align_up(o + (size_t)T * 4, 256);      // 8 bytes for each of at most T / 2 windows
  w.vis_list = o; o = align_up(o + (size_t)T * 4, 256);
  w.sim = o; o = align_up(o + nw * 8, 256);
  w.asum = o; o = align_up(o + nw * 8, 256);
  w.keep_idx = o; o = align_up(o + (size_t)T * 4, 256);
  w.kind = o; o = align_up(o + (size_t)T, 256);
  w.total = o;
  return w;
}
}  // namespace

extern "C" __attribute__((visibility("default"))) size_t fmmoe_prune_workspace_bytes(int64_t n_tokens, int32_t n_seq) {
  (void)n_seq;
  if (n_tokens < 0) return 0;
  return plan_prune(n_tokens).total + 256;
}

// The pruning pass in two phases: phase 1 (window scores, selection + compaction map)
// needs the routing probabilities and the mask only, phase 2 (row gather / merge) needs the rows.
// phases & 1 enqueues phase 1 on s_select, phases & 2 enqueues phase 2 on s_rows.  A caller that
// uses two streams orders phase 2 after phase 1 itself.
fmmoe_status fmmoe::prune_visual_phases(fmmoe_handle* h, const fmmoe_prune_params* p, const float* probs,
                                        int32_t n_experts, const float* attn, const void* x, int32_t dtype,
                                        int32_t hidden, const uint8_t* is_visual, const int64_t* seq_off,
                                        const int64_t* n_vis, const int64_t* n_retain, int32_t n_seq, void* x_out,
                                        uint8_t* is_visual_out, int32_t* keep_idx, uint8_t* kind,
                                        int64_t* out_seq_off, void* workspace, size_t workspace_bytes,
                                        int phases, cudaStream_t s_select, cudaStream_t s_rows, FinalizePrune* fused) {
  if (!h || !prune_params_ok(p) || !seq_off || !n_vis || !n_retain || !out_seq_off || n_seq < 0)
    return FMMOE_ERR_INVALID_ARG;
  if (n_experts < 1 || hidden < 1 || (dtype != FMMOE_F32 && dtype != FMMOE_BF16)) return FMMOE_ERR_INVALID_ARG;
  const int elem = dtype == FMMOE_BF16 ? 2 : 4;
  if ((hidden * elem) % 16 != 0) return FMMOE_ERR_UNSUPPORTED;
  int64_t max_nf = 0;
  out_seq_off[0] = 0;
  for (int b = 0; b < n_seq; ++b) {
    const int64_t L = seq_off[b + 1] - seq_off[b];
    if (L < 0 || n_vis[b] < 0 || n_vis[b] > L || n_retain[b] < 0) return FMMOE_ERR_INVALID_ARG;
    const int64_t kept = counts_for(n_vis[b], n_retain[b], p, nullptr, nullptr);
    out_seq_off[b + 1] = out_seq_off[b] + (L - n_vis[b]) + kept;
    if (n_vis[b] / p->window > max_nf) max_nf = n_vis[b] / p->window;
  }
  const int64_t T = n_seq ? seq_off[n_seq] : 0;
  if (n_seq && seq_off[0] != 0) return FMMOE_ERR_INVALID_ARG;
  if (T > 0x7fffffff) return FMMOE_ERR_UNSUPPORTED;
  if (T == 0) return FMMOE_OK;
  const int64_t T_out = out_seq_off[n_seq];
  if (!probs || !x || !is_visual || (T_out > 0 && !x_out)) return FMMOE_ERR_INVALID_ARG;
  if (x == x_out) return FMMOE_ERR_INVALID_ARG;
  if (((uintptr_t)x | (uintptr_t)x_out | (uintptr_t)probs) & 15) return FMMOE_ERR_INVALID_ARG;
  const PruneWs wp = plan_prune(T);
  if (!workspace || ((uintptr_t)workspace & 255) || workspace_bytes < wp.total) return FMMOE_ERR_WORKSPACE;
  if (max_nf > SEL_MAX_WINDOWS) return FMMOE_ERR_UNSUPPORTED;
  int64_t longest = 0;
  for (int b = 0; b < n_seq; ++b) longest = seq_off[b + 1] - seq_off[b] > longest ? seq_off[b + 1] - seq_off[b] : longest;
  const bool sel_small = longest <= SEL_SMALL_TOKENS && max_nf <= SEL_SMALL;
  const size_t sel_smem = (size_t)max_nf * (max_nf > SEL_THREADS ? 9 : 1);   // keys + action bytes of the longest sequence
  char* ws = static_cast<char*>(workspace);

  PruneDev a = {};
  a.probs = probs; a.attn = attn; a.x = x; a.is_visual = is_visual;
  a.E = n_experts; a.H = hidden; a.W = p->window; a.sim_mode = p->sim_mode; a.merge_mode = p->merge_mode;
  a.dtype = dtype; a.alpha = p->alpha;
  a.merges = reinterpret_cast<int2*>(ws + wp.merges); a.vis_list = reinterpret_cast<int32_t*>(ws + wp.vis_list);
  a.sim = reinterpret_cast<double*>(ws + wp.sim); a.asum = reinterpret_cast<double*>(ws + wp.asum);
  a.keep_idx_ws = reinterpret_cast<int32_t*>(ws + wp.keep_idx); a.kind_ws = reinterpret_cast<uint8_t*>(ws + wp.kind);
  a.x_out = x_out; a.is_visual_out = is_visual_out; a.keep_idx = keep_idx; a.kind = kind;
  a.status = h->d_status;
  a.late = !fused && prune_outputs_over_mask(is_visual, T, T_out, is_visual_out, keep_idx, kind);
  if (fused) {          // n_seq <= MAXS: one launch of each kernel
    a.pos = a.keep_idx_ws;
    fused->pos = a.pos; fused->x_out = x_out; fused->merges = a.merges; fused->vis_list = a.vis_list;
    fused->W = p->window; fused->merge_mode = p->merge_mode;
  }

  // select_kernel's dynamic shared-memory opt-in was raised once, in fmmoe_create

  int win_base = 0;
  for (int b0 = 0; b0 < n_seq; b0 += MAXS) {
    const int nb = n_seq - b0 < MAXS ? n_seq - b0 : MAXS;
    PruneSeqs sq = {};
    sq.n_seq = nb;
    sq.win_off[0] = win_base;
    for (int i = 0; i < nb; ++i) {
      const int b = b0 + i;
      int64_t m, d;
      counts_for(n_vis[b], n_retain[b], p, &m, &d);
      sq.n_vis[i] = (int)n_vis[b]; sq.m[i] = (int)m; sq.d[i] = (int)d;
      sq.win_off[i + 1] = sq.win_off[i] + (int)(n_vis[b] / p->window);
      sq.seq_off[i] = seq_off[b]; sq.out_off[i] = out_seq_off[b];
    }
    sq.seq_off[nb] = seq_off[b0 + nb]; sq.out_off[nb] = out_seq_off[b0 + nb];
    const int n_win = sq.win_off[nb] - win_base;
    // window ids inside a launch are relative to the launch's first window
    PruneSeqs rel = sq;
    for (int i = 0; i <= nb; ++i) rel.win_off[i] -= win_base;
    PruneDev al = a;
    al.sim = a.sim + win_base; al.asum = a.asum + win_base; al.merges = a.merges + win_base;
    int max_win = 0, n_merges = 0;
    for (int i = 0; i < nb; ++i) {
      const int w = rel.win_off[i + 1] - rel.win_off[i];
      max_win = w > max_win ? w : max_win;
      n_merges += rel.m[i];
    }
    if (fused) { fused->n_merges = n_merges; fused->sq = rel; }
    if (phases & 1) {
      cudaStream_t s = s_select;
      if (n_win > 0) {
        const unsigned ctas = (unsigned)((max_win + SC_WIN - 1) / SC_WIN);
        const ScoreKernel score = score_kernel(p->window, (int64_t)ctas * nb, h->sm_count, phases == 3);
        ProfScope ps(h, FMMOE_KERNEL_PRUNE_SCORE, s);
        for (int rep = 0; rep < ps.reps; ++rep, ++h->launches)
          FMMOE_CUDA_TRY(launch_pdl(score, dim3(ctas, nb), dim3(256), 0, s, 1, al, rel));
      }
      FMMOE_CUDA_TRY(cudaGetLastError());
      {
        PruneDev sel = al;
        if (al.late) { sel.is_visual_out = nullptr; sel.keep_idx = nullptr; sel.kind = nullptr; }
        ProfScope ps(h, FMMOE_KERNEL_PRUNE_SELECT, s);
        for (int rep = 0; rep < ps.reps; ++rep, ++h->launches)
          FMMOE_CUDA_TRY(launch_pdl(sel_small ? select_kernel<SEL_SMALL> : select_kernel<SEL_THREADS>, dim3(nb), dim3(sel_small ? SEL_SMALL : SEL_THREADS), sel_smem, s, 1, sel, rel));
      }
      FMMOE_CUDA_TRY(cudaGetLastError());
    }
    const long long rows = rel.out_off[nb] - rel.out_off[0];
    if ((phases & 2) && rows > 0) {
      cudaStream_t s = s_rows;
      const unsigned blocks = (unsigned)(n_merges + (rows + CP_ROWS - 1) / CP_ROWS);
      ProfScope ps(h, FMMOE_KERNEL_PRUNE_COMPACT, s);
      for (int rep = 0; rep < ps.reps; ++rep, ++h->launches) {
        if (dtype == FMMOE_BF16)
          FMMOE_CUDA_TRY(launch_pdl(compact_kernel<__nv_bfloat16>, dim3(blocks), dim3(256), 0, s, 1, al, rel, n_merges, (long long)rel.out_off[0], (long long)rows));
        else
          FMMOE_CUDA_TRY(launch_pdl(compact_kernel<float>, dim3(blocks), dim3(256), 0, s, 1, al, rel, n_merges, (long long)rel.out_off[0], (long long)rows));
      }
      FMMOE_CUDA_TRY(cudaGetLastError());
    }
    win_base += n_win;
  }
  return FMMOE_OK;
}

extern "C" __attribute__((visibility("default"))) fmmoe_status fmmoe_prune_visual(fmmoe_handle* h, const fmmoe_prune_params* p, const float* probs,
                                           int32_t n_experts, const float* attn, const void* x, int32_t dtype,
                                           int32_t hidden, const uint8_t* is_visual, const int64_t* seq_off,
                                           const int64_t* n_vis, const int64_t* n_retain, int32_t n_seq, void* x_out,
                                           uint8_t* is_visual_out, int32_t* keep_idx, uint8_t* kind,
                                           int64_t* out_seq_off, void* workspace, size_t workspace_bytes,
                                           void* cuda_stream) {
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  return prune_visual_phases(h, p, probs, n_experts, attn, x, dtype, hidden, is_visual, seq_off, n_vis, n_retain, n_seq,
                             x_out, is_visual_out, keep_idx, kind, out_seq_off, workspace, workspace_bytes, 3, s, s);
}

// ---------------------------------------------------------------------------------------
// fmmoe_prune_visual_static: the same pruning pass, with its scratch memory built into the
// library instead of supplied by the caller.
//
// Who needs it: code that must not ask the CUDA allocator for anything at the point where
// it prunes.  Examples are an inference server whose whole HBM budget was handed to another
// memory pool at start-up (a late cudaMalloc there fails or fragments the pool), and a
// latency-critical loop that cannot afford the device-wide synchronisation an allocation
// or a free may imply.  Such a caller still owns its inputs and outputs (they come from
// its pool); what it cannot do is size and carve out a workspace per call.
//
// The scratch is the file-scope device array below.  Every GPU on which the library is
// loaded holds these FMMOE_STATIC_PRUNE_SCRATCH_BYTES until the process exits.  In host
// code the array's name is only a stand-in for the symbol, never a device address, so the
// address is looked up with cudaGetSymbolAddress once per device (with that device
// current) and cached; kernels receive the looked-up pointer.
// ---------------------------------------------------------------------------------------
#define FMMOE_STATIC_PRUNE_SCRATCH_BYTES (768u * 1024u)
static __device__ __align__(256) unsigned char g_prune_scratch[FMMOE_STATIC_PRUNE_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
void* g_prune_scratch_addr[kMaxDevices] = {};     // device address of g_prune_scratch, per device
pthread_mutex_t g_prune_scratch_mu = PTHREAD_MUTEX_INITIALIZER;

// Device address of the scratch array on the CURRENT device (must be `device`); looked up on
// the first call for that device, cached afterwards.  Returns nullptr on failure.
void* static_scratch_for(int device) {
  if (device < 0 || device >= kMaxDevices) return nullptr;
  pthread_mutex_lock(&g_prune_scratch_mu);
  void* p = g_prune_scratch_addr[device];
  if (!p) {
    void* q = nullptr;
    if (cudaGetSymbolAddress(&q, g_prune_scratch) == cudaSuccess && q) {
      g_prune_scratch_addr[device] = q;
      p = q;
    }
  }
  pthread_mutex_unlock(&g_prune_scratch_mu);
  return p;
}
}  // namespace

// Called by fmmoe_create with the handle's device current.  Everything the pruning pass would
// otherwise do lazily on its first call happens here, at start-up, while the process can still
// obtain device memory: the module that holds the pruning kernels and the scratch array is loaded
// (under lazy module loading that is when the array and the kernel code are placed in device
// memory), the array's device address is looked up and cached, and select_kernel's dynamic
// shared-memory limit is raised once to what its longest sequence needs, so that no later call has to.
fmmoe_status fmmoe::prune_prepare(fmmoe_handle* h) {
  cudaFuncAttributes fa;
  for (const ScoreKernel k : kScore) FMMOE_CUDA_TRY(cudaFuncGetAttributes(&fa, k));
  for (const ScoreKernel k : kScoreFew) FMMOE_CUDA_TRY(cudaFuncGetAttributes(&fa, k));
  FMMOE_CUDA_TRY(cudaFuncGetAttributes(&fa, compact_kernel<__nv_bfloat16>));
  FMMOE_CUDA_TRY(cudaFuncGetAttributes(&fa, compact_kernel<float>));
  FMMOE_CUDA_TRY(cudaFuncGetAttributes(&fa, select_kernel<SEL_SMALL>));
  FMMOE_CUDA_TRY(cudaFuncGetAttributes(&fa, select_kernel<SEL_THREADS>));
  FMMOE_CUDA_TRY(cudaFuncSetAttribute(select_kernel<SEL_THREADS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SEL_MAX_WINDOWS * 9));
  if (!static_scratch_for(h->device)) return FMMOE_ERR_CUDA;
  return FMMOE_OK;
}

extern "C" __attribute__((visibility("default"))) fmmoe_status fmmoe_prune_visual_static(
    fmmoe_handle* h, const fmmoe_prune_params* p, const float* probs, int32_t n_experts, const float* attn,
    const void* x, int32_t dtype, int32_t hidden, const uint8_t* is_visual, const int64_t* seq_off,
    const int64_t* n_vis, const int64_t* n_retain, int32_t n_seq, void* x_out, uint8_t* is_visual_out,
    int32_t* keep_idx, uint8_t* kind, int64_t* out_seq_off, void* cuda_stream) {
  if (!h || !seq_off || n_seq < 0) return FMMOE_ERR_INVALID_ARG;
  const int64_t T = n_seq ? seq_off[n_seq] : 0;
  if (T < 0) return FMMOE_ERR_INVALID_ARG;
  // the limit is on the token count: refuse before touching the GPU
  if (T > FMMOE_STATIC_PRUNE_MAX_TOKENS) return FMMOE_ERR_TOO_LARGE;
  const size_t need = plan_prune(T).total;
  if (need > (size_t)FMMOE_STATIC_PRUNE_SCRATCH_BYTES) return FMMOE_ERR_TOO_LARGE;
  int cur = -1;
  if (cudaGetDevice(&cur) != cudaSuccess) return FMMOE_ERR_CUDA;
  if (cur != h->device) return FMMOE_ERR_INVALID_ARG;   // the handle's device must be current
  void* scratch = static_scratch_for(cur);
  if (!scratch) return FMMOE_ERR_CUDA;
  // Nothing in the scratch has to start at zero: a pass writes the vision lists, the
  // window scores and the compaction map before it reads them.  The one exception is a call
  // whose mask contradicts its n_vis: slots the pass then leaves unwritten hold the previous
  // call's values; the kernels range-check every index they take from the scratch, and the
  // mismatch is reported through the status word.
  return fmmoe_prune_visual(h, p, probs, n_experts, attn, x, dtype, hidden, is_visual, seq_off, n_vis, n_retain,
                            n_seq, x_out, is_visual_out, keep_idx, kind, out_seq_off, scratch,
                            (size_t)FMMOE_STATIC_PRUNE_SCRATCH_BYTES, cuda_stream);
}
