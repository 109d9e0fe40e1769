// The projection GEMMs for few tokens: 128 x BN tiles whose reduction is split over a thread-block cluster.
//
// A prompt of a few hundred tokens gives a projection fewer tiles than the chip has SMs (the gate of a
// 7B-shaped layer: 18 tiles of 128 x 256 at 333 tokens), and one tile walks the whole hidden dimension at
// what one SM takes in from L2 (~46 bytes a clock: 1,050 cycles per 64-deep k-block), whatever the number of
// tokens.  Here the S CTAs of a cluster take a share of the k-blocks each; their float32 accumulators
// go to their own shared memory (over the operand stages, free by then), and after a cluster barrier rank
// r adds up rows [r 128 / S, (r + 1) 128 / S) of the tile through distributed shared memory
// and hands them to the projection's epilogue, a warp per row.
//
// P (the projection) supplies: kExchangeUs (see choose_split); skip (a tile nobody wants); load_a / load_b (the TMA boxes of a k-block); prepare (work of the
// epilogue warps while the MMAs run); load_row (what the row's epilogue reads from memory, asked for together
// with the sums) and row (one finished row of BN columns: lane l has columns 4 l .. 4 l + 3 of every group of 128).
#pragma once
#include "ag_common.cuh"
#include "umma.cuh"

namespace ag {
namespace splitk {

using namespace umma;

constexpr int kBM = 128, kBK = 64, kThreads = 320;            // warps: TMA, MMA, 8 x epilogue
constexpr int kMaxSplit = 5;                                   // beyond, the exchange costs more than the k-blocks saved
template <int BN>
struct Cfg {
  static constexpr int kStages = BN == 256 ? 4 : 6;
  static constexpr int kABytes = kBM * kBK * 2;                // 16 KB
  static constexpr int kPanelBytes = kBK * 64 * 2;             // [64 k][64 n] = 8 KB
  static constexpr int kStageBytes = kABytes + (BN / 64) * kPanelBytes;
  static constexpr int kSmemBytes = kStages * kStageBytes + 1024 /*align*/ + 256 /*barriers*/;
  static_assert(kBM * BN * 4 <= kStages * kStageBytes, "the accumulator fits over the stages");
};
// Byte offset of 16-byte chunk `chunk` of row `row` of the float32 tile: XOR-ed with the row, so that neither
// the drain (a thread per row) nor the sums (a warp per row) meet bank conflicts.
template <int BN>
__device__ __forceinline__ uint32_t acc_off(int row, int chunk) { return (uint32_t)(row * BN * 4 + ((chunk ^ (row & 31)) << 4)); }

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}

__device__ __forceinline__ int ld_cluster_s32(uint32_t addr) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(addr));
  return v;
}

template <int BN, int splits, class P>
__global__ void __launch_bounds__(kThreads, 1)
gemm_splitk_kernel(const __grid_constant__ P p, int num_kb) {
  using C = Cfg<BN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + C::kStages * C::kStageBytes);
  uint64_t *empty = full + C::kStages;
  uint64_t *acc_full = empty + C::kStages;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(acc_full + 1);
  int *gave_up = reinterpret_cast<int *>(tmem_slot + 1);       // a wait of this CTA expired: its share of the sums is not there
  __shared__ typename P::Shared psh;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank(), tile = blockIdx.x / splits;
  const int kb_begin = rank * num_kb / splits, kb_end = (rank + 1) * num_kb / splits;    // never empty: splits <= num_kb

  if (p.skip(tile)) return;                          // the whole cluster
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(acc_full, 1);
    *gave_up = 0;
    fence_barrier_init();
    p.prefetch();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, BN);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem_acc = *tmem_slot;
  pdl_wait();                                        // set-up is done: what the kernel before wrote may be read
  pdl_launch_dependents();

  if (warp == 0) {
    if (lane == 0) {
      for (int kb = kb_begin; kb < kb_end; ++kb) {
        const int i = kb - kb_begin, s = i % C::kStages;
        if (!mbar_wait(&empty[s], ((i / C::kStages) & 1) ^ 1)) break;
        uint8_t *a = smem + s * C::kStageBytes;
        mbar_arrive_expect_tx(&full[s], C::kStageBytes);
        p.load_a(a, &full[s], tile, kb);
#pragma unroll
        for (int c = 0; c < BN / 64; ++c) p.load_b(a + C::kABytes + c * C::kPanelBytes, &full[s], tile, c, kb);
      }
    }
  } else if (warp == 1) {
    // every lane runs the control flow (operands stay warp-uniform); one elected lane issues
    constexpr uint32_t idesc = idesc_bf16_f32(kBM, BN, false, true);
    const uint64_t da0 = desc_kmajor_sw128(smem_u32(smem));
    const uint64_t db0 = desc_mnmajor_sw128(smem_u32(smem) + C::kABytes, C::kPanelBytes);
    const uint32_t a_lo0 = (uint32_t)da0, a_hi = (uint32_t)(da0 >> 32);
    const uint32_t b_lo0 = (uint32_t)db0, b_hi = (uint32_t)(db0 >> 32);
    for (int kb = kb_begin; kb < kb_end; ++kb) {
      const int i = kb - kb_begin, s = i % C::kStages;
      if (!mbar_wait(&full[s], (i / C::kStages) & 1)) {
        *gave_up = 1;
        break;
      }
      tc_fence_after_sync();
      const uint32_t a_lo = a_lo0 + ((s * C::kStageBytes) >> 4), b_lo = b_lo0 + ((s * C::kStageBytes) >> 4);
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < kBK / 16; ++k)
          mma_ss_lohi(tmem_acc, a_lo + ((k * 32) >> 4), a_hi, b_lo + ((k * 2048) >> 4), b_hi, idesc, (i | k) != 0);
        mma_commit(&empty[s]);     // frees the stage once these MMAs have read it
      }
      __syncwarp();
    }
    if (elect_one()) mma_commit(acc_full);   // accumulator complete (or unwinding)
    __syncwarp();
  } else {
    p.prepare(psh, tile, rank, splits);
    // all eight warps agree on whether the accumulator arrived
    if (!mbar_wait(acc_full, 0)) *gave_up = 1;
    named_barrier_sync(1, 256);
    if (*gave_up == 0) {
      tc_fence_after_sync();
      // warp w may touch TMEM lanes [32 * (w % 4), +32); warps 2..5 drain the first half of the columns, 6..9 the second
      const int quad = warp & 3, half = (warp - 2) >> 2, row = quad * 32 + lane;
#pragma unroll 1
      for (int c = half * (BN / 2); c < (half + 1) * (BN / 2); c += 32) {
        uint32_t r[32];
        tmem_ld_x32_sync(tmem_acc + ((uint32_t)(quad * 32) << 16) + c, r);
#pragma unroll
        for (int e = 0; e < 8; ++e)
          *reinterpret_cast<uint4 *>(smem + acc_off<BN>(row, (c >> 2) + e)) =
              make_uint4(r[4 * e], r[4 * e + 1], r[4 * e + 2], r[4 * e + 3]);
      }
    }
  }
  tc_fence_before_sync();
  __syncwarp();
  cluster_arrive_wait();                             // every CTA's accumulator lies in its shared memory
  if (warp >= 2 && *gave_up == 0) {
    // (A CTA that gave up holds operands where its sums should be: its tile is left unwritten by every rank.  Looked at
    // with the sums, so that nothing waits for it.)
    // Distributed shared memory answers late: kRows rows per warp in flight (up to 16 loads of 16 bytes per lane).
    constexpr int kChunks = BN / 128;                // 16-byte chunks (four columns) per lane
    constexpr int kRows = 16 / ((splits - 1) * kChunks);
    const uint32_t base = smem_u32(smem);
    const int row_end = (rank + 1) * kBM / splits;
    for (int row0 = rank * kBM / splits + (warp - 2) * kRows; row0 < row_end; row0 += 8 * kRows) {
      typename P::Row extra[kRows];
#pragma unroll
      for (int u = 0; u < kRows; ++u) extra[u] = p.load_row(tile, min(row0 + u, row_end - 1), lane * 4);
      // The CTA's own share comes from its shared memory, the others' in the order rank + 1, rank + 2, ...: no
      // CTA is asked by all at once, and a row's sum has a fixed order.
      float4 sum[kRows][kChunks], v[splits - 1][kRows][kChunks];
      int lost = 0;
#pragma unroll
      for (int i = 1; i < splits; ++i) {
        const int from = rank + i < splits ? rank + i : rank + i - splits;
        const uint32_t peer = mapa_shared(base, from);
        lost |= ld_cluster_s32(mapa_shared(smem_u32(gave_up), from));
#pragma unroll
        for (int u = 0; u < kRows; ++u)
#pragma unroll
          for (int c = 0; c < kChunks; ++c)
            v[i - 1][u][c] = ld_cluster_f4(peer + acc_off<BN>(min(row0 + u, row_end - 1), lane + 32 * c));
      }
#pragma unroll
      for (int u = 0; u < kRows; ++u)
#pragma unroll
        for (int c = 0; c < kChunks; ++c) {
          float4 t = *reinterpret_cast<const float4 *>(smem + acc_off<BN>(min(row0 + u, row_end - 1), lane + 32 * c));
#pragma unroll
          for (int i = 0; i < splits - 1; ++i) {
            t.x += v[i][u][c].x; t.y += v[i][u][c].y; t.z += v[i][u][c].z; t.w += v[i][u][c].w;
          }
          sum[u][c] = t;
        }
      if (lost != 0) break;
#pragma unroll
      for (int u = 0; u < kRows; ++u)
        if (row0 + u < row_end)
          p.row(psh, tile, row0 + u, lane * 4, reinterpret_cast<const float(&)[kChunks * 4]>(sum[u]), extra[u]);
    }
  }
  __syncwarp();
  cluster_arrive_wait();                             // nobody leaves while its accumulator may still be read
  if (warp == 1) tmem_dealloc(tmem_acc, BN);
}

// Host side: how many CTAs to split the reduction of `tiles` tiles over (1: not at all); cap[s] is how many clusters of s CTAs
// the device holds at once.  A round of tiles takes (us, fitted to the three projections at 100 .. 1500 tokens, hidden 512 ..
// 4096, 4 .. 32 heads, every number of CTAs) 0.33 per k-block of 256 columns (0.25 of 128) and 5 beside them; split, 0.45
// (0.34) per k-block, and exchange_us for set-up, the two cluster barriers and the exchange.  Split in 1 | 2 | 3 | 4 | 5:
//   output projection of 100 tokens, 64 k-blocks   26.2 | 21.9 | 18.2 | 15.0 | 14.8     300 tokens, 16   10.4 | 12.1 | 11.8 | 9.9 | 10.3
//   key/value projection of 100 tokens, 64   26.4 | 26.3 | 22.0 | 18.0 | 31.1     500 tokens, 9 heads, 32   13.9 | 17.7 | 26.0 | 31.5 | 30.3
template <int BN>
int choose_split(long long tiles, int num_kb, const int *cap, double exchange_us) {
  constexpr double kKbUs = BN == 256 ? 0.33 : 0.25;
  int best = 1;
  double best_t = 1e30;
  for (int s = 1; s <= kMaxSplit; ++s) {
    if (cap[s] <= 0 || (s > 1 && num_kb / s < 2)) continue;
    const double rounds = (double)((tiles + cap[s] - 1) / cap[s]);
    const double t = rounds * (s == 1 ? kKbUs * num_kb + 5 : 1.36 * kKbUs * ((num_kb + s - 1) / s) + exchange_us);
    if (t < 0.97 * best_t) { best_t = t; best = s; }
  }
  return best;
}

template <int BN, class P>
cudaLaunchConfig_t splitk_config(int ctas, int splits, cudaStream_t st, cudaLaunchAttribute *attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = Cfg<BN>::kSmemBytes;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = splits; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1] = pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cfg;
}

template <int BN, class P>
using Kernel = void (*)(const P, int);
template <int BN, class P>
Kernel<BN, P> kernel_of(int splits) {
  switch (splits) {
    case 2: return gemm_splitk_kernel<BN, 2, P>;
    case 3: return gemm_splitk_kernel<BN, 3, P>;
    case 4: return gemm_splitk_kernel<BN, 4, P>;
    default: return gemm_splitk_kernel<BN, 5, P>;
  }
}

// Clusters of every size the current device holds at once (asked for once per device and kernel); [1]: SMs.
template <int BN, class P>
int splitk_capacity(const int **out) {
  static int cap[64][kMaxSplit + 1];
  static int ready[64];
  int dev = 0;
  AG_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return AG_ERR_UNSUPPORTED;
  if (!__atomic_load_n(&ready[dev], __ATOMIC_ACQUIRE)) {
    AG_CUDA_TRY(cudaDeviceGetAttribute(&cap[dev][1], cudaDevAttrMultiProcessorCount, dev));
    for (int s = 2; s <= kMaxSplit; ++s) {
      auto kern = kernel_of<BN, P>(s);
      AG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<BN>::kSmemBytes));
      cudaLaunchAttribute attr[2];
      cudaLaunchConfig_t cfg = splitk_config<BN, P>(s, s, nullptr, attr);
      int n = 0;
      AG_CUDA_TRY(cudaOccupancyMaxActiveClusters(&n, kern, &cfg));
      cap[dev][s] = n;                               // the same values whichever thread writes them
    }
    __atomic_store_n(&ready[dev], 1, __ATOMIC_RELEASE);
  }
  *out = cap[dev];
  return AG_OK;
}

template <int BN, class P>
int launch_splitk(const P &p, long long tiles, int num_kb, int splits, cudaStream_t st) {
  auto kern = kernel_of<BN, P>(splits);
  AG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<BN>::kSmemBytes));
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = splitk_config<BN, P>((int)(tiles * splits), splits, st, attr);
  AG_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, p, num_kb));
  return AG_OK;
}

}  // namespace splitk
}  // namespace ag
