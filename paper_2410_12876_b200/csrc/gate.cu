// The Attention-Gate pass (Sec. 3.3): AG(X) = G(MHA'(X), tau), Eq. 3 / Eq. 4,
// with the optional constant gamma inside the Sigmoid (Sec. 3.5).
//
//   1. projection   [Q' | K' | V'] = X [Wq_g | Wk_g | Wv_g]   (tcgen05 GEMM for bf16, else CUDA cores)
//   2. MHA'         H'_g = Softmax(Q'_g K'_g^T / sqrt(d'_k)) V'_g  (tcgen05 on two or three bf16
//                   parts per value for bf16 layers with h' d'_k a multiple of 128, else float32 on CUDA cores)
//   3. output layer    s = [H'_1 .. H'_h'] Wo_g;  flag = s + gamma > logit(tau)
//                   (gate_out_kernel; on the tensor-core path fused into the merge of MHA's split-K partials)
//
// The scores decide a hard threshold, so everything after the (exact) products
// of the input elements is kept in float32: a flag can then differ from an
// infinitely precise evaluation only for scores within ~1e-5 of the threshold.
#include <math.h>

#include "ag_common.cuh"
#include "attn_simt.cuh"

namespace ag {

constexpr int kGemmBK = 32;

// C[M, 3*GD] (float32) = A[M, Kd] * [W0 | W1 | W2], each W [Kd, GD] row-major: the CUDA-core form.
// One CTA of 256 threads = BT x BT outputs (64: 4 x 4 per thread; 32: 2 x 2, for few tokens, so that more SMs
// work).  k-blocks of 32 arrive by asynchronous copies, the next one while one is worked on; A is read four k
// at a time.  Bound by arithmetic and, at few tokens, by the length of the chain over K: 16 k at a time with
// scalar loads behind the barrier took 16.9 us for 128 x 256 x 384.
template <typename T, int BT>
__global__ void __launch_bounds__(256)
gate_proj_kernel(const T *A, const T *W0, const T *W1, const T *W2, float *C, int M, int Kd, int GD) {
  constexpr int TM = BT / 16, AP = kGemmBK + 4, kEpl = Elem<T>::kPerVec;
  __shared__ __align__(16) float As[2][BT][AP];
  __shared__ __align__(16) float Ws[2][kGemmBK][BT];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * BT;
  const int n0 = blockIdx.x * BT;                // column in the packed [3*GD] output
  const int which = n0 / GD, nw = n0 % GD;       // GD is a multiple of 64: a tile never straddles
  const T *W = which == 0 ? W0 : (which == 1 ? W1 : W2);
  // (No early trigger of MHA': its CTAs, set up beside this kernel's, crowded onto few SMs; 95 -> 40 us for the pass of 500
  // tokens of two 64-wide gate heads, 224 -> 135 for 1,000 of three with bf16 inputs.)
  // k-block kb -> buffer kb & 1; rows past M are clamped (never stored), k past Kd is zero (Kd is a multiple of 8)
  auto load_block = [&](int kb) {
    const int k0 = kb * kGemmBK, buf = kb & 1;
    for (int x = tid; x < BT * kGemmBK / kEpl; x += 256) {
      const int ar = x / (kGemmBK / kEpl), ak = x % (kGemmBK / kEpl) * kEpl;
      const int wr = x / (BT / kEpl), wc = x % (BT / kEpl) * kEpl;
      const bool a_in = k0 + ak < Kd, w_in = k0 + wr < Kd;
      const T *from_a = A + (size_t)min(m0 + ar, M - 1) * Kd + (a_in ? k0 + ak : 0);
      const T *from_w = W + (size_t)(w_in ? k0 + wr : 0) * GD + nw + wc;
      if constexpr (sizeof(T) == 4) {
        cp_async16_zfill((uint32_t)__cvta_generic_to_shared(&As[buf][ar][ak]), from_a, a_in ? 16 : 0);
        cp_async16_zfill((uint32_t)__cvta_generic_to_shared(&Ws[buf][wr][wc]), from_w, w_in ? 16 : 0);
      } else {
        float fa[kEpl], fw[kEpl];
        Elem<T>::unpack(a_in ? ld128(from_a) : make_uint4(0u, 0u, 0u, 0u), fa);
        Elem<T>::unpack(w_in ? ld128(from_w) : make_uint4(0u, 0u, 0u, 0u), fw);
#pragma unroll
        for (int e = 0; e < kEpl; ++e) { As[buf][ar][ak + e] = fa[e]; Ws[buf][wr][wc + e] = fw[e]; }
      }
    }
    cp_async_commit();
  };
  float acc[TM][TM];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) acc[i][j] = 0.f;

  const int n_blocks = (Kd + kGemmBK - 1) / kGemmBK;
  load_block(0);
  for (int kb = 0; kb < n_blocks; ++kb) {
    if (kb + 1 < n_blocks) {
      load_block(kb + 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const int buf = kb & 1;
#pragma unroll
    for (int k = 0; k < kGemmBK; k += 4) {
      float4 av[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) av[i] = *reinterpret_cast<const float4 *>(&As[buf][ty * TM + i][k]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float w[TM];
#pragma unroll
        for (int j = 0; j < TM; ++j) w[j] = Ws[buf][k + u][tx * TM + j];
#pragma unroll
        for (int i = 0; i < TM; ++i) {
          const float x = u == 0 ? av[i].x : u == 1 ? av[i].y : u == 2 ? av[i].z : av[i].w;
#pragma unroll
          for (int j = 0; j < TM; ++j) acc[i][j] = fmaf(x, w[j], acc[i][j]);
        }
      }
    }
    __syncthreads();                             // the buffer may be refilled
  }
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int row = m0 + ty * TM + i;
    if (row < M) {
#pragma unroll
      for (int j = 0; j < TM; ++j) C[(size_t)row * 3 * GD + n0 + tx * TM + j] = acc[i][j];
    }
  }
}

// s = [H'_1 .. H'_h'] Wo_g and the threshold of Eq. 4.  One CTA = kTokens tokens, one
// warp = kTokens / 4 of them, lane = head (in rounds of 32 heads).  The rows of H and a
// [GD][32] slice of Wo are staged in shared memory: per step of the reduction a
// warp reads one conflict-free row of Wo and a broadcast value of H per token.  4 tokens where 16 would leave
// most SMs without a CTA.
constexpr int kOutThreads = 128;
template <typename T, int kOutTokens>
__global__ void __launch_bounds__(kOutThreads)
gate_out_kernel(const float *H, const T *__restrict__ Wo,
                const float *__restrict__ gamma, float logit_tau, int B, int n, int GD, int h,
                const int32_t *__restrict__ seq_lens, float *__restrict__ scores, uint8_t *__restrict__ flags) {
  constexpr int kPer = kOutTokens / 4;           // tokens per warp
  extern __shared__ __align__(16) unsigned char sh_raw[];
  float *Hs = reinterpret_cast<float *>(sh_raw);                       // [16][GD]
  T *Ws = reinterpret_cast<T *>(sh_raw + sizeof(float) * kOutTokens * GD);   // [GD][32]
  const int tiles_per_seq = (n + kOutTokens - 1) / kOutTokens;
  const int b = blockIdx.x / tiles_per_seq, t0 = (blockIdx.x % tiles_per_seq) * kOutTokens;
  const int nt = min(kOutTokens, n - t0);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  pdl_wait();
  pdl_launch_dependents();
  const float *Hg = H + ((size_t)b * n + t0) * GD;                     // rows are contiguous
  for (int x = threadIdx.x; x < kOutTokens * GD; x += kOutThreads) Hs[x] = x < nt * GD ? Hg[x] : 0.f;
  for (int i0 = 0; i0 < h; i0 += 32) {
    __syncthreads();
    for (int x = threadIdx.x; x < GD * 32; x += kOutThreads) {
      const int c = x >> 5, i = i0 + (x & 31);
      Ws[x] = i < h ? Wo[(size_t)c * h + i] : T(0.f);
    }
    __syncthreads();
    float acc[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) acc[q] = 0.f;
    const float *hr = Hs + warp * kPer * GD;
#pragma unroll 8
    for (int c = 0; c < GD; ++c) {
      const float w = Elem<T>::load(Ws + c * 32 + lane);
#pragma unroll
      for (int q = 0; q < kPer; ++q) acc[q] = fmaf(hr[q * GD + c], w, acc[q]);
    }
    const int i = i0 + lane;
    if (i < h) {
      const float gm = gamma ? gamma[i] : 0.f;
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const int tt = warp * kPer + q;
        if (tt < nt) {
          const size_t o = ((size_t)b * h + i) * n + t0 + tt;
          const bool padding = seq_lens && t0 + tt >= seq_lens[b];
          if (scores) scores[o] = acc[q];
          flags[o] = !padding && (acc[q] + gm) > logit_tau ? 1 : 0;
        }
      }
    }
  }
}

size_t gate_workspace_bytes(const ag_layer_desc &d) {
  const size_t rows = (size_t)d.batch * d.seq, GD = (size_t)d.gate_heads * d.gate_head_dim;
  // [Q' | K' | V'] (float32, or its bf16 parts), then H' (CUDA-core path) or the split-K
  // partials of MHA' (tensor-core path, where H' stays on chip)
  if (d.dtype == AG_BF16 && gate_attn_tc_supported(d))
    return align_up(rows * 3 * GD * 2 * gate_attn_parts(d), 256) + gate_attn_partial_bytes(d);
  return align_up(rows * 3 * GD * sizeof(float), 256) + align_up(rows * GD * sizeof(float), 256);
}

template <typename T>
static int run_gate(const ag_layer_desc &d, const void *X, const void *Wq, const void *Wk,
                    const void *Wv, const void *Wo, const float *gamma, float *scores,
                    uint8_t *flags, void *ws, cudaStream_t st) {
  const int M = d.batch * d.seq, GD = d.gate_heads * d.gate_head_dim, Dg = d.gate_head_dim;
  float *qkv = static_cast<float *>(ws);
  float *hcat = reinterpret_cast<float *>(static_cast<char *>(ws) +
                                          align_up((size_t)M * 3 * GD * sizeof(float), 256));
  const float logit_tau = (float)log((double)d.tau / (1.0 - (double)d.tau));
  if (sizeof(T) == 2 && gate_attn_tc_supported(d)) {
    // tensor-core path: projections as bf16 parts, MHA' on tcgen05 with a product per pair of parts that matters.
    // Padding is projected only as far as MHA' reads it, to the end of the 128-token tile a sequence ends in.
    const int parts = gate_attn_parts(d);
    int rc = launch_gate_proj_tc(X, Wq, Wk, Wv, ws, parts, M, d.hidden, GD, d.seq_lens, d.seq, st);
    if (rc) return rc;
    void *partials = static_cast<char *>(ws) + align_up((size_t)M * 3 * GD * 2 * parts, 256);   // H' stays on chip
    // the merge of the split-K partials carries the output layer and the threshold with it
    return launch_gate_attn_tc(d, ws, partials, Wo, gamma, logit_tau, scores, flags, st);
  } else {
    if (sizeof(T) == 2 && gate_proj_tc_supported(d.hidden, GD)) {
      int rc = launch_gate_proj_tc(X, Wq, Wk, Wv, qkv, 0, M, d.hidden, GD, nullptr, d.seq, st);
      if (rc) return rc;
    } else {
      auto p = [](const void *x) { return static_cast<const T *>(x); };
      // 64 x 64 outputs per CTA, or 32 x 32 where that leaves half of the SMs without a CTA (pass of 48 tiles of 64: 41.4 us,
      // 39.7 at 32; of 120: 58.7, 68.6; of 144: 109, 135)
      if ((long long)(3 * GD / 64) * ((M + 63) / 64) >= 148 / 2)
        gate_proj_kernel<T, 64><<<dim3(3 * GD / 64, (M + 63) / 64), 256, 0, st>>>(p(X), p(Wq), p(Wk), p(Wv), qkv, M, d.hidden, GD);
      else
        gate_proj_kernel<T, 32><<<dim3(3 * GD / 32, (M + 31) / 32), 256, 0, st>>>(p(X), p(Wq), p(Wk), p(Wv), qkv, M, d.hidden, GD);
      AG_LAUNCH_CHECK();
    }
    SimtAttnArgs a{};
    a.Q = qkv; a.K = qkv + GD; a.V = qkv + 2 * GD; a.O = hcat;
    a.n = d.seq; a.inner = d.gate_heads;
    a.q_batch = a.k_batch = a.v_batch = (long long)d.seq * 3 * GD;
    a.q_inner = a.k_inner = a.v_inner = Dg;
    a.q_row = a.k_row = a.v_row = 3 * GD;
    a.o_batch = (long long)d.seq * GD; a.o_inner = Dg; a.o_row = GD;
    a.scale_log2 = (float)(1.4426950408889634 / sqrt((double)Dg));
    a.seq_lens = d.seq_lens;
    const int problems = d.batch * d.gate_heads;
    int rc;
    if (Dg == 64)
      rc = d.gate_causal ? launch_simt_attn<float, float, 64, kGateCausal>(a, problems, st)
                         : launch_simt_attn<float, float, 64, kGateFull>(a, problems, st);
    else
      rc = d.gate_causal ? launch_simt_attn<float, float, 128, kGateCausal>(a, problems, st)
                         : launch_simt_attn<float, float, 128, kGateFull>(a, problems, st);
    if (rc) return rc;
  }

  const int tokens = d.batch * d.seq <= 16 * 148 ? 4 : 16;
  const size_t out_smem = sizeof(float) * (size_t)tokens * GD + sizeof(T) * (size_t)GD * 32;
  auto out_kern = tokens == 4 ? gate_out_kernel<T, 4> : gate_out_kernel<T, 16>;
  AG_CUDA_TRY(cudaFuncSetAttribute(out_kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)out_smem));
  const int blocks = d.batch * ((d.seq + tokens - 1) / tokens);
  return launch_pdl(out_kern, dim3(blocks), dim3(kOutThreads), out_smem, st, hcat, static_cast<const T *>(Wo), gamma,
                    logit_tau, d.batch, d.seq, GD, kv_heads_of(d), d.seq_lens, scores, flags);
}

int launch_gate(const ag_layer_desc &d, const void *X, const void *Wq, const void *Wk,
                const void *Wv, const void *Wo, const float *gamma, float *scores,
                uint8_t *flags, void *ws, cudaStream_t st) {
  if (d.dtype == AG_F32) return run_gate<float>(d, X, Wq, Wk, Wv, Wo, gamma, scores, flags, ws, st);
  return run_gate<__nv_bfloat16>(d, X, Wq, Wk, Wv, Wo, gamma, scores, flags, ws, st);
}

}  // namespace ag
