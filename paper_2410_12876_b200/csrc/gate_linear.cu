// The local gate of Sec. 3.4 ("Local or global?", ablation setting (5)): MHA' is
// replaced by one linear layer, s = X W_lin, followed by the threshold of Eq. 4
// (gamma of Sec. 3.5 inside the Sigmoid).  A token's flag depends on its own
// hidden state only.
//
// s is a skinny contraction, [B n, d] x [d, h] with h a few dozen columns: the
// kernel is bound by reading X once.  bf16 layers run on the tensor cores
// (products of bf16 inputs are exact in the float32 accumulator): one CTA owns
// 128 tokens and a slice of d; the CTAs of a thread-block cluster split d among
// them so that enough CTAs stream X, and then the heads: each adds its heads'
// partial accumulators in rank order through distributed shared memory (a fixed
// order: results do not vary from run to run), thresholds and writes.
//
// A CTA alone takes 16 KB of X and 8 KB of W per trip; three CTAs of three stages share an SM, so that one's set-up, first
// trip and exchange lie under the others' streams.  us for 100 | 2000 | 4096 | 2 x 3001 | 11,000 | 20,000 tokens of 4096, 32 heads:
//   one CTA of six stages, all heads added up by one rank      11.1 | 21.7 | 14.7 | 16.4 | 24.8 | 49.6
//   the heads shared among the ranks, one CTA of eight stages  6.5 | 12.2 | 11.7 | 16.2 | 25.9 | 53.0
//   two of four stages                                         6.5 | 7.9 | 10.9 | 14.8 | 23.6 | 38.7
//   three of three                                             6.4 | 7.9 | 11.2 | 13.6 | 21.7 | 34.6
//   with a loop of as many ranks as there are                  5.7 | 7.3 | 10.9 | 13.4 | 20.0 | 31.4   (5.2 TB/s)
//   A = X      [B n, d]  row-major -> K-major operand, 128-byte swizzled rows
//   B = W_lin  [d, h]    row-major -> MN-major operand: one panel of [64 k][64 n],
//                                     columns past h filled with zeros by TMA
// Other layers (float32, h > 64, odd strides) take a CUDA-core kernel.
#include <cooperative_groups.h>
#include <math.h>

#include "ag_common.cuh"
#include "launch_rules.cuh"
#include "umma.cuh"

namespace ag {

using namespace umma;
namespace cg = cooperative_groups;

constexpr int kGlBM = 128, kGlBK = 64, kGlThreads = 192, kGlStages = 3;
constexpr int kGlCtasPerSm = 3;
constexpr int kGlABytes = kGlBM * kGlBK * 2;              // 16 KB
constexpr int kGlBBytes = kGlBK * 64 * 2;                 // one panel [64 k][64 n] = 8 KB
constexpr int kGlStageBytes = kGlABytes + kGlBBytes;
constexpr int kGlMaxN = 64;                               // heads the tensor-core kernel serves
// The partial accumulator of a CTA, [col][row], lies over the stages once every MMA has read them.
static_assert(kGlBM * kGlMaxN * 4 <= kGlStages * kGlStageBytes, "partial sums");
constexpr int kGlSmemBytes = kGlStages * kGlStageBytes + 1024 /*align*/ + 256 /*barriers*/;
constexpr uint32_t kGlTmemCols = 64;

struct GateLinearArgs {
  const int32_t *seq_lens;   // [B] or NULL: tokens past seq_lens[b] are padding (flag 0)
  const float *gamma;
  float *scores;
  uint8_t *flags;
  int M, n, h, kb_total;               // tokens, sequence length, heads, 64-wide k blocks
  float logit_tau;
};

// N: MMA width, heads rounded up to 32.  kRanks: CTAs of a tile's cluster.
template <int N, int kRanks>
__global__ void __launch_bounds__(kGlThreads, kGlCtasPerSm)
gate_linear_tc_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                      const GateLinearArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  float *part = reinterpret_cast<float *>(smem);          // [N][128]
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + kGlStages * kGlStageBytes);
  uint64_t *empty = full + kGlStages;
  uint64_t *acc_full = empty + kGlStages;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_full + 1);

  cg::cluster_group cluster = cg::this_cluster();
  const int rank = kRanks == 1 ? 0 : (int)cluster.block_rank();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * kGlBM;
  const int kb_begin = rank * a.kb_total / kRanks, kb_end = (rank + 1) * a.kb_total / kRanks;
  // a tile that holds padding only: no scores to compute, flags 0
  const int num_kb = padding_rows(a.seq_lens, a.n, m0, min(m0 + kGlBM, a.M), 1) ? 0 : kb_end - kb_begin;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kGlStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(acc_full, 1);
    fence_barrier_init();
    prefetch_tensormap(&tmX);
    prefetch_tensormap(&tmW);
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, kGlTmemCols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_acc = *tmem_slot;
  pdl_wait();                                        // set-up is done: what the kernel before wrote may be read

  if (warp == 0) {
    if (lane == 0) {
      for (int kb = 0; kb < num_kb; ++kb) {
        const int s = kb % kGlStages;
        const uint32_t ph = (kb / kGlStages) & 1;
        if (!mbar_wait(&empty[s], ph ^ 1)) break;
        uint8_t *sa = smem + s * kGlStageBytes, *sb = sa + kGlABytes;
        mbar_arrive_expect_tx(&full[s], kGlStageBytes);
        tma_load_2d(sa, &tmX, &full[s], (kb_begin + kb) * kGlBK, m0);
        tma_load_2d(sb, &tmW, &full[s], 0, (kb_begin + kb) * kGlBK);
      }
    }
  } else if (warp == 1) {
    // every lane runs the control flow (operands stay warp-uniform); one elected lane issues
    constexpr uint32_t idesc = idesc_bf16_f32(kGlBM, N, false, true);
    const uint64_t da0 = desc_kmajor_sw128(smem_u32(smem));
    const uint64_t db0 = desc_mnmajor_sw128(smem_u32(smem) + kGlABytes, kGlBBytes);
    const uint32_t a_lo0 = (uint32_t)da0, a_hi = (uint32_t)(da0 >> 32);
    const uint32_t b_lo0 = (uint32_t)db0, b_hi = (uint32_t)(db0 >> 32);
    bool ok = true;
    for (int kb = 0; kb < num_kb && ok; ++kb) {
      const int s = kb % kGlStages;
      const uint32_t ph = (kb / kGlStages) & 1;
      ok = mbar_wait(&full[s], ph);
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t a_lo = a_lo0 + ((s * kGlStageBytes) >> 4), b_lo = b_lo0 + ((s * kGlStageBytes) >> 4);
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < kGlBK / 16; ++k)
          mma_ss_lohi(tmem_acc, a_lo + ((k * 32) >> 4), a_hi, b_lo + ((k * 2048) >> 4), b_hi, idesc, (kb | k) != 0);
        mma_commit(&empty[s]);
      }
      __syncwarp();
    }
    if (elect_one()) mma_commit(acc_full);   // accumulator complete (or unwinding)
    __syncwarp();
  } else {
    // thread = token row
    const int quad = warp & 3, r_in = quad * 32 + lane;
    const int tok = m0 + r_in;
    const int b = tok / a.n, t = tok % a.n;
    const bool valid = tok < a.M;
    const bool padding = valid && a.seq_lens && t >= a.seq_lens[b];
    auto write = [&](int i, float s) {
      const size_t o = ((size_t)b * a.h + i) * a.n + t;        // lanes = consecutive tokens: coalesced
      if (a.scores) a.scores[o] = s;
      a.flags[o] = !padding && (s + (a.gamma ? a.gamma[i] : 0.f)) > a.logit_tau ? 1 : 0;
    };
    const bool ok = mbar_wait(acc_full, 0);
    tc_fence_after_sync();
#pragma unroll
    for (int c = 0; c < N; c += 32) {
      uint32_t r[32];
      if (ok && num_kb > 0) {
        tmem_ld_x32_sync(tmem_acc + ((uint32_t)(quad * 32) << 16) + c, r);
      } else {
#pragma unroll
        for (int e = 0; e < 32; ++e) r[e] = 0u;
      }
#pragma unroll
      for (int e = 0; e < 32; ++e) {
        if constexpr (kRanks > 1) part[(c + e) * kGlBM + r_in] = __uint_as_float(r[e]);     // the CTA's partial sums, [col][row]
        else if (valid && c + e < a.h) write(c + e, __uint_as_float(r[e]));
      }
    }
    if constexpr (kRanks > 1) {
      cluster.sync();                   // every CTA's partial sums are in its shared memory
      // Each CTA adds up, thresholds and writes its share of the heads: rank, rank + kRanks, ...
      // (All eight ranks' places gone over whatever kRanks: 2 us of a call with one or two CTAs to a tile.)
      constexpr int kAtOnce = kRanks == 2 ? 8 : 4;             // heads: 16 or 32 values per thread in flight
      const float *p[kRanks];
#pragma unroll
      for (int rk = 0; rk < kRanks; ++rk) p[rk] = cluster.map_shared_rank(part, rk) + r_in;
#pragma unroll 1
      for (int i0 = rank; valid && i0 < a.h; i0 += kAtOnce * kRanks) {
        float x[kAtOnce][kRanks];
#pragma unroll
        for (int u = 0; u < kAtOnce; ++u)
#pragma unroll
          for (int rk = 0; rk < kRanks; ++rk) x[u][rk] = i0 + u * kRanks < a.h ? p[rk][(i0 + u * kRanks) * kGlBM] : 0.f;
#pragma unroll
        for (int u = 0; u < kAtOnce; ++u) {
          float s = 0.f;
#pragma unroll
          for (int rk = 0; rk < kRanks; ++rk) s += x[u][rk];   // rank order: the sum does not depend on timing
          if (i0 + u * kRanks < a.h) write(i0 + u * kRanks, s);
        }
      }
    }
  }
  if constexpr (kRanks > 1) {
    __syncwarp();
    if (warp < 2) cluster.sync();       // (the one above)
    cluster.sync();                     // partial sums stay alive until every CTA has read them
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_acc, kGlTmemCols);
}

// CUDA-core form: one warp per token, lanes stride over d, heads in registers eight at a time.
template <typename T>
__global__ void __launch_bounds__(256)
gate_linear_simt_kernel(const T *__restrict__ X, const T *__restrict__ W, const float *__restrict__ gamma,
                        float logit_tau, int M, int n, int d, int h, const int32_t *__restrict__ seq_lens,
                        float *__restrict__ scores, uint8_t *__restrict__ flags) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tok = blockIdx.x * 8 + warp;
  if (tok >= M) return;
  const int b = tok / n, t = tok % n;
  const T *x = X + (size_t)tok * d;
  for (int i0 = 0; i0 < h; i0 += 8) {
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    for (int k = lane; k < d; k += 32) {
      const float xv = Elem<T>::load(x + k);
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (i0 + e < h) acc[e] = fmaf(xv, Elem<T>::load(W + (size_t)k * h + i0 + e), acc[e]);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], off);
    }
    if (lane == 0) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int i = i0 + e;
        if (i < h) {
          const size_t o = ((size_t)b * h + i) * n + t;
          if (scores) scores[o] = acc[e];
          flags[o] = !(seq_lens && t >= seq_lens[b]) && (acc[e] + (gamma ? gamma[i] : 0.f)) > logit_tau ? 1 : 0;
        }
      }
    }
  }
}

// How many clusters of a size the device holds at once is asked of a kernel of the same threads and shared memory: one that
// allocates tensor memory is answered for as if a CTA took all of an SM's.
__global__ void __launch_bounds__(kGlThreads, kGlCtasPerSm) gate_linear_place_kernel() {}

static cudaLaunchConfig_t gate_linear_config(int ranks, int m_tiles, cudaStream_t st, cudaLaunchAttribute *attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ranks, m_tiles);
  cfg.blockDim = dim3(kGlThreads);
  cfg.dynamicSmemBytes = kGlSmemBytes;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ranks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1] = pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

// Asked for once per thread and context.
static int gate_linear_places(GateLinearPlaces *out) {
  struct Answer { unsigned long long context; GateLinearPlaces places; };
  static thread_local Answer known[8] = {};
  const unsigned long long context = current_context();
  Answer &a = known[context % 8];
  if (context == 0 || a.context != context) {
    AG_CUDA_TRY(cudaFuncSetAttribute(gate_linear_place_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGlSmemBytes));
    for (int i = 0; i < kGlSplits; ++i) {
      cudaLaunchAttribute attr[2];
      const cudaLaunchConfig_t cfg = gate_linear_config(1 << i, 1, nullptr, attr);
      AG_CUDA_TRY(cudaOccupancyMaxActiveClusters(&a.places.clusters[i], gate_linear_place_kernel, &cfg));
    }
    a.context = context;
  }
  *out = a.places;
  return AG_OK;
}

template <int N, int kRanks>
static int launch_gate_linear_tc(const CUtensorMap &tmX, const CUtensorMap &tmW, const GateLinearArgs &a, int m_tiles, cudaStream_t st) {
  auto kern = gate_linear_tc_kernel<N, kRanks>;
  AG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kGlSmemBytes));
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = gate_linear_config(kRanks, m_tiles, st, attr);
  AG_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, tmX, tmW, a));
  return AG_OK;
}

template <int N>
static int run_gate_linear_tc(const ag_layer_desc &d, const void *X, const void *W, const GateLinearArgs &a, cudaStream_t st) {
  CUtensorMap tmX, tmW;
  int rc = make_tmap_2d_bf16(&tmX, X, a.M, d.hidden, (uint64_t)d.hidden * 2, kGlBM, kGlBK);
  if (rc) return rc;
  rc = make_tmap_2d_bf16(&tmW, W, d.hidden, kv_heads_of(d), (uint64_t)kv_heads_of(d) * 2, kGlBK, 64);
  if (rc) return rc;
  GateLinearPlaces places;
  if ((rc = gate_linear_places(&places))) return rc;
  const int m_tiles = (a.M + kGlBM - 1) / kGlBM;
  switch (gate_linear_split(m_tiles, a.kb_total, a.h, places)) {
    case 1: return launch_gate_linear_tc<N, 1>(tmX, tmW, a, m_tiles, st);
    case 2: return launch_gate_linear_tc<N, 2>(tmX, tmW, a, m_tiles, st);
    case 4: return launch_gate_linear_tc<N, 4>(tmX, tmW, a, m_tiles, st);
    default: return launch_gate_linear_tc<N, 8>(tmX, tmW, a, m_tiles, st);
  }
}

int launch_gate_linear(const ag_layer_desc &d, const void *X, const void *W, const float *gamma,
                       float *scores, uint8_t *flags, cudaStream_t st) {
  GateLinearArgs a;
  a.seq_lens = d.seq_lens; a.gamma = gamma; a.scores = scores; a.flags = flags;
  a.M = d.batch * d.seq; a.n = d.seq; a.h = kv_heads_of(d);
  a.kb_total = (d.hidden + kGlBK - 1) / kGlBK;
  a.logit_tau = (float)log((double)d.tau / (1.0 - (double)d.tau));
  const bool tc = d.dtype == AG_BF16 && kv_heads_of(d) <= kGlMaxN && kv_heads_of(d) % 8 == 0 && d.hidden % 8 == 0 &&
                  (int64_t)d.batch * d.seq < ((int64_t)1 << 31) - kGlBM && (a.M + kGlBM - 1) / kGlBM <= 65535;
  if (tc) {
    if (kv_heads_of(d) <= 32) return run_gate_linear_tc<32>(d, X, W, a, st);
    return run_gate_linear_tc<64>(d, X, W, a, st);
  }
  const int blocks = (a.M + 7) / 8;
  if (d.dtype == AG_F32)
    gate_linear_simt_kernel<float><<<blocks, 256, 0, st>>>(static_cast<const float *>(X), static_cast<const float *>(W),
                                                          gamma, a.logit_tau, a.M, a.n, d.hidden, kv_heads_of(d), d.seq_lens, scores, flags);
  else
    gate_linear_simt_kernel<__nv_bfloat16><<<blocks, 256, 0, st>>>(
        static_cast<const __nv_bfloat16 *>(X), static_cast<const __nv_bfloat16 *>(W), gamma, a.logit_tau, a.M, a.n,
        d.hidden, kv_heads_of(d), d.seq_lens, scores, flags);
  AG_LAUNCH_CHECK();
  return AG_OK;
}

int gate_linear_wait_timeouts() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, umma::g_wait_expired, sizeof(int)) != cudaSuccess) return -1;
  return v;
}

}  // namespace ag
