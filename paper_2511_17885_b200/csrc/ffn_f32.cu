// Expert FFNs in fp32 (Eq. 4 with SwiGLU experts) for fp32 layers.  Plain FMA on
// CUDA cores: TF32 tensor cores would not meet an fp32 tolerance.  Same grouping,
// same two GEMMs and the same combine as the tensor-core path.  A CTA forms 32 rows x 64 weight rows (GEMM-1: 32 gate
// and the same 32 up features; GEMM-2: 64 hidden columns).
// fp32 layers are small, so a CTA's time is the latency of its walk along the contraction.  Hence four groups of 128
// threads that each take a quarter of every 128-element k-slab (their sums are added at the end), the next slab on
// its way by cp.async while this one is multiplied, 4 x 4 outputs a thread read as 16-byte vectors, two multiply-adds an instruction
// (8 loads for 32 of them), and in GEMM-2 with the atomic combine CTAs that share out the contraction: each adds its share to the token's
// row, in any order, so that a row may differ in its last bits from call to call whatever the number of experts (FMMOE_FLAG_DETERMINISTIC: one CTA, a fixed
// order).  The shares of a tile added up in order by a cluster of its CTAs, one add a row: the small layer 28.6 -> 30.2 us, with a shared expert 46.8 -> 50.2.
// The small layer (H 256, 8 experts of 512, 256 tokens) in a graph of layers: GEMM-1 12.5 us, GEMM-2 7.6 (before the spills below went), against 12.7 and 21.3 with the
// contraction in one CTA and one multiply-add an instruction.  In the atomic combine without the residual the sums are the output
// itself (api.cu): 2-3 us and a launch for the pass that copied them.
#include "internal.h"
#include "ptx.cuh"

namespace fmmoe {

constexpr int F_BM = F32_BLOCK_M;   // 32
constexpr int F_BN = 64;            // weight rows per CTA
constexpr int F_KG = 4;             // k-groups
constexpr int F_KS = 32;            // k elements of a group per slab
constexpr int F_BK = F_KG * F_KS;
constexpr int F_LD = F_BK + 4;      // row pitch in shared memory: 16-byte reads of eight rows hit distinct banks
constexpr int F_LDR = F_BN + 16;    // row pitch of the partial sums
constexpr int F_THREADS = F_KG * 128;
constexpr int F_ROWS = F_BM + F_BN;
constexpr int F_STAGE_FLOATS = F_ROWS * F_LD;
constexpr int F_SMEM_BYTES = 2 * F_STAGE_FLOATS * 4;
static_assert(F_KG * F_BM * F_LDR <= 2 * F_STAGE_FLOATS, "partial sums overlay the slabs");
static_assert(F_BK == 128 && F_ROWS % (F_THREADS / 32) == 0, "a warp loads one row of a slab at a time");

struct F32Params {
  const MTile* mtiles; const int32_t* n_mtiles;   // routed M-tiles (NULL for the shared launch)
  int mt_per_shared; long long T;                 // shared launch: tiles per shared expert
  int K;                                          // contraction length
  int N;                                          // output columns per group
  const float* a;                                 // MODE 0: x [T, K];  MODE 1: act [rows, K]
  const int32_t* row_token;                       // routed: token of each grouped row
  const float* row_gate;
  const float* b0; const float* b1;               // [groups, N, K] (b1: up projection, MODE 0)
  float* out;                                     // MODE 0: act [rows, N]; MODE 1 det: y [rows, N]
  float* acc;                                     // MODE 1 atomic: [T, N]
  int deterministic;
  int k_slabs;                                    // slabs of a CTA (MODE 1 atomic: blockIdx.z takes its share of the contraction)
};

template <int MODE>
__global__ void __launch_bounds__(F_THREADS, 2) ffn_f32_kernel(const F32Params p) {
  extern __shared__ __align__(16) float f_smem[];   // two slabs of [F_BM rows of A | F_BN weight rows][F_LD]
  pdl_launch_dependents();
  pdl_wait();
  const bool routed = p.mtiles != nullptr;
  int group, row0, rows;
  if (routed) {
    const int n = *p.n_mtiles;
    const int4 m4 = *reinterpret_cast<const int4*>(p.mtiles + blockIdx.x);      // asked for together: the list is as long as the grid
    if ((int)blockIdx.x >= n) return;
    const MTile m = {m4.x, m4.y, m4.z, m4.w};
    group = m.group; row0 = m.row0; rows = m.rows;
  } else {
    group = blockIdx.x / p.mt_per_shared;
    row0 = (blockIdx.x - group * p.mt_per_shared) * F_BM;
    const long long left = p.T - row0;
    rows = left < F_BM ? (int)left : F_BM;
  }
  constexpr int NC = MODE == 0 ? F_BN / 2 : F_BN;   // output columns per CTA
  const int n0 = blockIdx.y * NC;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // output row index in the grouped space (shared experts: group * T + token)
  const long long out_base = routed ? row0 : (long long)group * p.T + row0;
  // rows of a slab that this warp loads (one 512-byte row at a time, 16 bytes a lane): F_BM / WARPS of A, then the weights'
  constexpr int WARPS = F_THREADS / 32, RPW = F_ROWS / WARPS, RPA = F_BM / WARPS;
  static_assert(F_BM % WARPS == 0, "a warp's first rows are A's");
  const float* src[RPA];
#pragma unroll
  for (int i = 0; i < RPA; ++i) {
    const int r = i * WARPS + warp;
    long long ar = -1;
    if (r < rows) ar = MODE == 0 ? (routed ? (long long)p.row_token[row0 + r] : row0 + r) : out_base + r;
    src[i] = ar >= 0 ? p.a + ar * p.K + lane * 4 : nullptr;
  }
  // Weight row i of a warp (from RPA on): row n0 + w of its matrix, w growing with i (GEMM-1: the gate rows, then the same up rows).  One
  // offset for all of them: with a pointer a row the kernels spilled 36-40 bytes; the small layer of 256 tokens 28.7 -> 27.7 us, with a shared
  // expert 46.9 -> 44.9, 128 experts of 256 (H 1,024) 260.8 -> 256.5.
  const long long w0 = ((long long)group * p.N + n0 + warp) * p.K + lane * 4;
  const int n_w = p.N - n0 - warp;       // rows from the warp's first on
  const uint32_t smem0 = smem_u32(f_smem);
  auto load_slab = [&](int k0, int stage) {
    const bool k_ok = k0 + lane * 4 < p.K;          // K is a multiple of 4
#pragma unroll
    for (int j = 0; j < RPW; ++j) {
      const int i = (j + RPA) % RPW;                // the weights first: they do not wait for the rows' tokens
      const float* at;
      if (i < RPA) {
        at = src[i];
      } else {
        const int c = (i - RPA) * WARPS, w = MODE == 0 ? c % NC : c;
        at = w < n_w ? (MODE == 0 && c >= NC ? p.b1 : p.b0) + w0 + (long long)w * p.K : nullptr;
      }
      const bool ok = k_ok && at != nullptr;
      const uint32_t dst = smem0 + 4u * (uint32_t)(stage * F_STAGE_FLOATS + (i * WARPS + warp) * F_LD + lane * 4);
      cp_async_16_or_zero(dst, ok ? static_cast<const void*>(at + k0) : static_cast<const void*>(p.a), ok);
    }
    cp_async_commit();
  };
  const int kg = tid >> 7, tx = tid & 15, ty = (tid >> 4) & 7;   // outputs: rows ty + 8 i, weight rows tx + 16 j
  float2 acc[4][4] = {};      // sums over the even and the odd k
  const int s0 = MODE == 1 ? (int)blockIdx.z * p.k_slabs : 0, n_slabs = min((p.K + F_BK - 1) / F_BK - s0, p.k_slabs);
  load_slab(s0 * F_BK, 0);
  for (int s = 0; s < n_slabs; ++s) {
    if (s + 1 < n_slabs) { load_slab((s0 + s + 1) * F_BK, (s + 1) & 1); cp_async_wait_all_but<1>(); }
    else cp_async_wait_all_but<0>();
    __syncthreads();
    const float* As = f_smem + (s & 1) * F_STAGE_FLOATS + kg * F_KS;
    const float* Bs = As + F_BM * F_LD;
#pragma unroll 1
    for (int k = 0; k < F_KS; k += 4) {
      float4 av[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) av[i] = *reinterpret_cast<const float4*>(As + (ty + 8 * i) * F_LD + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 bv = *reinterpret_cast<const float4*>(Bs + (tx + 16 * j) * F_LD + k);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          fma2(acc[i][j], make_float2(av[i].x, av[i].y), make_float2(bv.x, bv.y));
          fma2(acc[i][j], make_float2(av[i].z, av[i].w), make_float2(bv.z, bv.w));
        }
      }
    }
    __syncthreads();
  }
  // the groups' sums, added in group order
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) f_smem[(kg * F_BM + ty + 8 * i) * F_LDR + tx + 16 * j] = acc[i][j].x + acc[i][j].y;
  __syncthreads();
  auto total = [&](int r, int c) {
    float v = f_smem[r * F_LDR + c];
#pragma unroll
    for (int g = 1; g < F_KG; ++g) v += f_smem[(g * F_BM + r) * F_LDR + c];
    return v;
  };
  if (MODE == 0) {
    for (int o = tid; o < F_BM * NC; o += F_THREADS) {
      const int r = o / NC, c = o % NC;
      if (r >= rows || n0 + c >= p.N) continue;
      const float g = total(r, c);
      p.out[(out_base + r) * p.N + n0 + c] = g / (1.f + expf(-g)) * total(r, c + NC);
    }
  } else {
    for (int o = tid; o < F_BM * NC / 4; o += F_THREADS) {
      const int r = o / (NC / 4), c = o % (NC / 4) * 4;
      if (r >= rows || n0 + c >= p.N) continue;          // N is a multiple of 4
      float4 v = make_float4(total(r, c), total(r, c + 1), total(r, c + 2), total(r, c + 3));
      if (p.deterministic) {
        *reinterpret_cast<float4*>(p.out + (out_base + r) * p.N + n0 + c) = v;
      } else {
        const long long tok = routed ? p.row_token[row0 + r] : row0 + r;
        const float gate = routed ? p.row_gate[row0 + r] : 1.f;
        v.x *= gate; v.y *= gate; v.z *= gate; v.w *= gate;
        atomicAdd(reinterpret_cast<float4*>(p.acc + tok * p.N + n0 + c), v);
      }
    }
  }
}

fmmoe_status launch_ffn_f32(fmmoe_handle* h, const FfnArgs& a, cudaStream_t s) {
  const fmmoe_layer_desc& d = *a.d;
  const int H = d.hidden, I = d.inter, Ns = d.n_shared, Is = d.shared_inter;
  if (a.T == 0) return FMMOE_OK;
  const int mtps = (int)((a.T + F_BM - 1) / F_BM);
  auto slabs_of = [](int K) { return (K + F_BK - 1) / F_BK; };
  // GEMM-2 with the atomic combine: the contraction is shared out where its tiles leave SMs idle (two CTAs fit one), a slab at least a
  // CTA.  `tiles`: M-tiles there are likely to be.
  auto split_k = [&](int K, long long tiles, int N) {
    const long long ctas = tiles * ((N + F_BN - 1) / F_BN), most = a.deterministic ? 1 : slabs_of(K);
    long long ks = (4ll * h->sm_count) / (ctas > 0 ? ctas : 1);
    ks = ks < 1 ? 1 : ks > most ? most : ks;
    return (int)((slabs_of(K) + ks - 1) / ks);      // slabs a CTA
  };
  if (!h->f32_attr_set) {
    FMMOE_CUDA_TRY(cudaFuncSetAttribute(ffn_f32_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, F_SMEM_BYTES));
    FMMOE_CUDA_TRY(cudaFuncSetAttribute(ffn_f32_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, F_SMEM_BYTES));
    h->f32_attr_set = true;
  }
  // routed GEMM-1
  F32Params p = {};
  p.mtiles = a.mtiles; p.n_mtiles = a.n_mtiles; p.T = a.T;
  p.K = H; p.N = I; p.a = static_cast<const float*>(a.x);
  p.row_token = a.row_token; p.row_gate = a.row_gate;
  p.b0 = static_cast<const float*>(a.w->w_gate); p.b1 = static_cast<const float*>(a.w->w_up);
  p.out = static_cast<float*>(a.act); p.k_slabs = slabs_of(H);
  if (a.max_mtiles > 0) {
    { ProfScope prof_(h, FMMOE_KERNEL_GEMM1, s); FMMOE_CUDA_TRY(launch_pdl(ffn_f32_kernel<0>, dim3(a.max_mtiles, (I + F_BN / 2 - 1) / (F_BN / 2)), dim3(F_THREADS), F_SMEM_BYTES, s, 1, p)); }
    FMMOE_CUDA_TRY(cudaGetLastError());
    // routed GEMM-2
    F32Params q = p;
    q.K = I; q.N = H; q.a = static_cast<const float*>(a.act);
    q.b0 = static_cast<const float*>(a.w->w_down); q.b1 = nullptr;
    q.out = a.y; q.acc = a.acc; q.deterministic = a.deterministic;
    q.k_slabs = split_k(I, (a.p_max < d.n_experts ? a.p_max : d.n_experts) + a.p_max / F_BM, H);
    { ProfScope prof_(h, FMMOE_KERNEL_GEMM2, s); FMMOE_CUDA_TRY(launch_pdl(ffn_f32_kernel<1>, dim3(a.max_mtiles, (H + F_BN - 1) / F_BN, (slabs_of(I) + q.k_slabs - 1) / q.k_slabs), dim3(F_THREADS), F_SMEM_BYTES, s, 1, q)); }
    FMMOE_CUDA_TRY(cudaGetLastError());
    h->launches += 2;
  }
  if (Ns) {
    F32Params ps = {};
    ps.mt_per_shared = mtps; ps.T = a.T; ps.K = H; ps.N = Is; ps.a = static_cast<const float*>(a.x);
    ps.b0 = static_cast<const float*>(a.w->ws_gate); ps.b1 = static_cast<const float*>(a.w->ws_up);
    ps.out = static_cast<float*>(a.act_sh); ps.k_slabs = slabs_of(H);
    { ProfScope prof_(h, FMMOE_KERNEL_GEMM1, s); FMMOE_CUDA_TRY(launch_pdl(ffn_f32_kernel<0>, dim3(Ns * mtps, (Is + F_BN / 2 - 1) / (F_BN / 2)), dim3(F_THREADS), F_SMEM_BYTES, s, 1, ps)); }
    FMMOE_CUDA_TRY(cudaGetLastError());
    F32Params qs = ps;
    qs.K = Is; qs.N = H; qs.a = static_cast<const float*>(a.act_sh);
    qs.b0 = static_cast<const float*>(a.w->ws_down); qs.b1 = nullptr;
    qs.out = a.ysh; qs.acc = a.acc; qs.deterministic = a.deterministic;
    qs.k_slabs = split_k(Is, (long long)Ns * mtps, H);
    { ProfScope prof_(h, FMMOE_KERNEL_GEMM2, s); FMMOE_CUDA_TRY(launch_pdl(ffn_f32_kernel<1>, dim3(Ns * mtps, (H + F_BN - 1) / F_BN, (slabs_of(Is) + qs.k_slabs - 1) / qs.k_slabs), dim3(F_THREADS), F_SMEM_BYTES, s, 1, qs)); }
    FMMOE_CUDA_TRY(cudaGetLastError());
    h->launches += 2;
  }
  return FMMOE_OK;
}

}  // namespace fmmoe
