// float32 CUDA-core attention used where the tensor-core path does not apply:
// the fp32 layer (tcgen05 has no true-fp32 MMA) and the fp32 internals of the
// gate (MHA' of Sec. 3.3 evaluated on float32 Q', K', V').
//
// One CTA = BM (64, 32 or 16) query rows x one problem (sequence, head); keys are visited in
// tiles of 64 with an online softmax, whatever BM, so a row's result does not depend on it.  Thread
// (tx, ty) of 16 x 16 holds rows ty * BM / 16 .. and keys tx, tx + 16, tx + 32, tx + 48 of a tile.  K and V
// lie row-major in shared memory (rows of D + 4 floats: the 16-byte reads of eight lanes fall into
// different banks) and arrive by 16-byte asynchronous copies: the next K while the weighted sum runs, V
// while the scores are computed.  Inner loops read 16 bytes of every operand per four steps.
// Few query tiles (a short prompt) get small BM, so that more SMs work: 128 tokens of 4 heads of 64 (8 CTAs at
// BM = 64) 25 -> 10.6 us.
// Row j sees the first bound(j) rows of the key array, where bound is
//   kGateCausal : j + 1            (lower-triangular mask inside MHA')
//   kGateFull   : n                (every token sees the whole sequence)
//   kPrefill    : prefix[s, j]     (retained tokens before j, read from the
//                                   compacted cache) plus the self term (k_j,
//                                   v_j) from the dense K, V: Eq. 5.
#pragma once
#include "ag_common.cuh"
#include "mma_sync.cuh"

namespace ag {

enum SimtAttnMode { kGateCausal = 0, kGateFull = 1, kPrefill = 2 };

struct SimtAttnArgs {
  const void *Q, *K, *V;      // kPrefill: K, V are the DENSE tensors (self term)
  void *O;
  int n;                      // query rows per problem
  int inner;                  // problems per batch element (h' or h)
  int kv_group;               // kPrefill: query heads per key/value head (0 or 1 = one each)
  long long q_batch, q_inner, q_row;   // element strides
  long long k_batch, k_inner, k_row;   // gate: K/V rows inside the packed projection
  long long v_batch, v_inner, v_row;
  long long o_batch, o_inner, o_row;
  float scale_log2;
  // kPrefill only
  const void *k_rows, *v_rows;         // compacted cache pools
  const int64_t *row_off;
  const int32_t *prefix;               // [problems, n + 1]
  const int32_t *len;                  // [problems] valid rows of each slab: a row bound never exceeds it
  float *lse;                          // NULL, or [problems, n]: m + log2(l) of every row
  // [batch] tokens each sequence has (the rest is padding), or NULL = n: the keys of kGateFull, and
  // the query tiles kPrefill has to compute
  const int32_t *seq_lens;
};

constexpr int kSimtBN = 64, kSimtThreads = 256;

template <int D, int BM>
constexpr size_t simt_attn_smem_bytes() {
  return sizeof(float) * ((size_t)(BM + kSimtBN) * (D + 4) + (size_t)kSimtBN * D + (size_t)BM * (kSimtBN + 4));
}

template <typename TIn, typename TOut, int D, int MODE, int BM>
__global__ void __launch_bounds__(kSimtThreads)
simt_attn_kernel(const SimtAttnArgs a) {
  extern __shared__ __align__(16) float smem[];
  constexpr int QP = D + 4, PP = kSimtBN + 4;     // row pitches
  float *Qs = smem;                               // [BM][QP]
  float *Ks = Qs + BM * QP;                       // [BN][QP]
  float *Vs = Ks + kSimtBN * QP;                  // [BN][D]
  float *Ps = Vs + kSimtBN * D;                   // [BM][PP]
  constexpr int RM = BM / 16;                     // rows per thread
  constexpr int kEpl = Elem<TIn>::kPerVec;
  constexpr int kVecPerRow = D / kEpl;
  constexpr int kOC = D / 64;                     // float4 column groups per thread

  const int prob = blockIdx.y;
  const int b = prob / a.inner, i = prob % a.inner;
  const int j0 = (gridDim.x - 1 - blockIdx.x) * BM;   // the tiles with the most keys first
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;

  pdl_wait();
  pdl_launch_dependents();
  const TIn *Qp = static_cast<const TIn *>(a.Q) + b * a.q_batch + i * a.q_inner;
  // grouped-query attention: query head i reads key/value head ik, cache slab prob_kv
  const int group = a.kv_group > 1 ? a.kv_group : 1;
  const int ik = i / group, prob_kv = b * (a.inner / group) + ik;
  const TIn *Kd = static_cast<const TIn *>(a.K) + b * a.k_batch + ik * a.k_inner;
  const TIn *Vd = static_cast<const TIn *>(a.V) + b * a.v_batch + ik * a.v_inner;
  const TIn *Kp = Kd, *Vp = Vd;
  long long kp_row = a.k_row, vp_row = a.v_row;
  if (MODE == kPrefill) {
    Kp = static_cast<const TIn *>(a.k_rows) + a.row_off[prob_kv] * (long long)D;
    Vp = static_cast<const TIn *>(a.v_rows) + a.row_off[prob_kv] * (long long)D;
    kp_row = D; vp_row = D;
  }
  const int32_t *pre = MODE == kPrefill ? a.prefix + (size_t)prob_kv * (a.n + 1) : nullptr;
  // a slab that overflowed at compaction holds no rows (len = 0) although its prefix counts are
  // full: its queries then see themselves only, and no read leaves the slab
  const int slab_len = MODE == kPrefill ? a.len[prob_kv] : 0;
  const int n_keys = (MODE == kGateFull && a.seq_lens) ? a.seq_lens[prob / a.inner] : a.n;
  // prefill: a query tile past its sequence's end holds padding only (outputs unspecified): nothing to do
  if (MODE == kPrefill && a.seq_lens && j0 >= a.seq_lens[prob / a.inner]) return;

  // rows r0 .. of src -> shared rows of `pitch` floats; rows past `last` are clamped (masked below, or never stored)
  auto load_rows = [&](float *dst, int pitch, const TIn *src, long long row_stride, int r0, int count, int last) {
    for (int x = tid; x < count * kVecPerRow; x += kSimtThreads) {
      const int r = x / kVecPerRow, c = x % kVecPerRow;
      const TIn *from = src + min(r0 + r, last) * row_stride + c * kEpl;
      float *to = dst + r * pitch + c * kEpl;
      if constexpr (sizeof(TIn) == 4) {
        cp_async16((uint32_t)__cvta_generic_to_shared(to), from);
      } else {
        float f[kEpl];
        Elem<TIn>::unpack(ld128(from), f);
#pragma unroll
        for (int e = 0; e < kEpl; ++e) to[e] = f[e];
      }
    }
    cp_async_commit();
  };

  int bound[RM];
  bool valid[RM];
#pragma unroll
  for (int r = 0; r < RM; ++r) {
    const int j = j0 + ty * RM + r;
    valid[r] = j < a.n;
    const int jc = min(j, a.n - 1);
    bound[r] = MODE == kGateCausal ? jc + 1 : (MODE == kGateFull ? n_keys : min(pre[jc], slab_len));
    if (!valid[r]) bound[r] = 0;
  }
  const int j_last = min(j0 + BM, a.n) - 1;
  const int max_bound = MODE == kGateCausal ? j_last + 1 : (MODE == kGateFull ? n_keys : min(pre[j_last], slab_len));
  const int n_tiles = (max_bound + kSimtBN - 1) / kSimtBN;
  const int t_last = max_bound - 1;                 // rows past it are masked for every query
  load_rows(Qs, QP, Qp, a.q_row, j0, BM, a.n - 1);
  if (n_tiles > 0) {
    load_rows(Ks, QP, Kp, kp_row, 0, kSimtBN, t_last);
    load_rows(Vs, D, Vp, vp_row, 0, kSimtBN, t_last);
  }

  float m[RM], l[RM], o[RM][kOC][4];
#pragma unroll
  for (int r = 0; r < RM; ++r) {
    m[r] = -INFINITY; l[r] = 0.f;
#pragma unroll
    for (int c = 0; c < kOC; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[r][c][e] = 0.f;
  }

  if (MODE == kPrefill) {
    // self term: the diagonal of Eq. 5 seeds the running softmax (m = s_jj, l = 1, o = v_j)
#pragma unroll
    for (int r = 0; r < RM; ++r) {
      const int j = min(j0 + ty * RM + r, a.n - 1);
      float acc = 0.f;
#pragma unroll
      for (int d = 0; d < D; d += 16)
        acc = fmaf(Elem<TIn>::load(Qp + j * a.q_row + d + tx), Elem<TIn>::load(Kd + j * a.k_row + d + tx), acc);
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
      m[r] = acc * a.scale_log2;
      l[r] = 1.f;
#pragma unroll
      for (int c = 0; c < kOC; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[r][c][e] = Elem<TIn>::load(Vd + j * a.v_row + c * 64 + tx * 4 + e);
    }
  }

  for (int kt = 0; kt < n_tiles; ++kt) {
    const int t0 = kt * kSimtBN;
    cp_async_wait<1>();                             // Q and this K (this thread's pieces)
    __syncthreads();                                // ... and everybody's
    float s[RM][4];
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) s[r][c] = 0.f;
#pragma unroll 4
    for (int d = 0; d < D; d += 4) {
      float4 qv[RM];
#pragma unroll
      for (int r = 0; r < RM; ++r) qv[r] = *reinterpret_cast<const float4 *>(&Qs[(ty * RM + r) * QP + d]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float4 kv = *reinterpret_cast<const float4 *>(&Ks[(tx + 16 * c) * QP + d]);
#pragma unroll
        for (int r = 0; r < RM; ++r) {
          s[r][c] = fmaf(qv[r].x, kv.x, s[r][c]);
          s[r][c] = fmaf(qv[r].y, kv.y, s[r][c]);
          s[r][c] = fmaf(qv[r].z, kv.z, s[r][c]);
          s[r][c] = fmaf(qv[r].w, kv.w, s[r][c]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < RM; ++r) {
      float mx = -INFINITY;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const bool vis = t0 + tx + 16 * c < bound[r];
        s[r][c] = vis ? s[r][c] * a.scale_log2 : -INFINITY;
        mx = fmaxf(mx, s[r][c]);
      }
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      const float m_new = fmaxf(m[r], mx);
      const float alpha = (m_new == -INFINITY) ? 1.f : exp2f(m[r] - m_new);
      float rs = 0.f;
      float p[4];
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        p[c] = (s[r][c] == -INFINITY) ? 0.f : exp2f(s[r][c] - m_new);
        rs += p[c];
      }
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) rs += __shfl_xor_sync(0xffffffffu, rs, off);
      l[r] = l[r] * alpha + rs;
      m[r] = m_new;
#pragma unroll
      for (int c = 0; c < kOC; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[r][c][e] *= alpha;
#pragma unroll
      for (int c = 0; c < 4; ++c) Ps[(ty * RM + r) * PP + tx + 16 * c] = p[c];
    }
    cp_async_wait<0>();                             // this V
    __syncthreads();                                // V and P complete; K has been read
    if (kt + 1 < n_tiles) load_rows(Ks, QP, Kp, kp_row, t0 + kSimtBN, kSimtBN, t_last);
#pragma unroll 4
    for (int t = 0; t < kSimtBN; t += 4) {
      float4 pv[RM];
#pragma unroll
      for (int r = 0; r < RM; ++r) pv[r] = *reinterpret_cast<const float4 *>(&Ps[(ty * RM + r) * PP + t]);
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int c = 0; c < kOC; ++c) {
          const float4 vv = *reinterpret_cast<const float4 *>(&Vs[(t + u) * D + c * 64 + tx * 4]);
#pragma unroll
          for (int r = 0; r < RM; ++r) {
            const float w = u == 0 ? pv[r].x : u == 1 ? pv[r].y : u == 2 ? pv[r].z : pv[r].w;
            o[r][c][0] = fmaf(w, vv.x, o[r][c][0]);
            o[r][c][1] = fmaf(w, vv.y, o[r][c][1]);
            o[r][c][2] = fmaf(w, vv.z, o[r][c][2]);
            o[r][c][3] = fmaf(w, vv.w, o[r][c][3]);
          }
        }
    }
    if (kt + 1 < n_tiles) {
      __syncthreads();                              // V and P have been read
      load_rows(Vs, D, Vp, vp_row, t0 + kSimtBN, kSimtBN, t_last);
    }
  }
  cp_async_wait<0>();                               // (Q alone, where there was no tile)

  TOut *Op = static_cast<TOut *>(a.O) + b * a.o_batch + i * a.o_inner;
#pragma unroll
  for (int r = 0; r < RM; ++r) {
    if (!valid[r]) continue;
    const int j = j0 + ty * RM + r;
    const float inv = 1.f / l[r];
    if (MODE == kPrefill && a.lse != nullptr && tx == 0) a.lse[(size_t)prob * a.n + j] = m[r] + log2f(l[r]);
#pragma unroll
    for (int c = 0; c < kOC; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        Elem<TOut>::store(Op + j * a.o_row + c * 64 + tx * 4 + e, o[r][c][e] * inv);
  }
}

template <typename TIn, typename TOut, int D, int MODE, int BM>
int launch_simt_attn_bm(const SimtAttnArgs &a, int problems, cudaStream_t st) {
  constexpr size_t smem = simt_attn_smem_bytes<D, BM>();
  auto kern = simt_attn_kernel<TIn, TOut, D, MODE, BM>;
  AG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  return launch_pdl(kern, dim3((a.n + BM - 1) / BM, problems), dim3(kSimtThreads), smem, st, a);
}

// BM by the number of CTAs it gives.  A key tile costs a CTA about 4,500, 5,000 or 9,000 cycles at BM = 16, 32, 64
// (D = 128: the first two are bound by shared-memory reads, the last by FMA issue), so 32 is nearly as
// quick per CTA as 16 and 64 the cheapest per row only once every SM has two.
template <typename TIn, typename TOut, int D, int MODE>
int launch_simt_attn(const SimtAttnArgs &a, int problems, cudaStream_t st) {
  constexpr long long kSms = 148;
  auto ctas = [&](int bm) { return (long long)((a.n + bm - 1) / bm) * problems; };
  if (ctas(64) >= 2 * kSms) return launch_simt_attn_bm<TIn, TOut, D, MODE, 64>(a, problems, st);
  if (ctas(32) >= kSms / 2) return launch_simt_attn_bm<TIn, TOut, D, MODE, 32>(a, problems, st);
  return launch_simt_attn_bm<TIn, TOut, D, MODE, 16>(a, problems, st);
}

}  // namespace ag
