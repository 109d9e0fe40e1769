// Core of decode attention on warp-level MMAs: rows [r_begin, r_end) of one key/value slab against
// the G <= 16 query vectors that read it (G query heads of a group, or one head), streamed through
// shared memory.  Used by the chunk pass of grouped-query decode and by the cluster form of decode.
//
// m16n8k16 bf16 MMAs (a tcgen05 tile needs 64 rows or more): the contraction is bound by memory, and what the tensor
// cores buy is fewer instructions per row, not FLOP/s.  Both products are turned, S^T = K Q^T and O^T = V^T P^T, so that
// the keys, then the dims, are the 16 rows of an MMA and the query heads its 8 columns: half the MMAs and half
// the accumulators of the form with the (mostly empty) 16 query rows; S^T becomes the second operand of the
// weighted sum by an 8 x 8 transpose between registers (movmatrix).
// The weights P enter the weighted sum as two bf16 parts each (one would cost the outputs a third of their accuracy:
// error against float64 of 72 .. 256 slabs 2.2e-3 with one part, 1.65e-3, the rounding of the outputs, with two).  Up to
// four heads the second part is free: columns 4 .. 7 of the MMAs repeat the heads, with the low parts as their weights,
// and the two halves are added at the end.  More heads take a second MMA per block.
// Rows go global -> shared by 16-byte cp.async in tiles of 64 rows (K and V; the next tile is in flight while one is
// worked on); each of the four warps fetches and owns 16 rows of every tile and keeps its own running softmax, so the
// warps wait for nobody until their (m, l, o) triples end in shared memory, where gq_combine() merges them.
// Measured: chunk pass of 32 sequences x 8 slabs of 1600 .. 7400 rows, four heads each, 104.5 -> 101.8 us per step.
#pragma once
#include "ag_common.cuh"
#include "mma_sync.cuh"

namespace ag {

constexpr int kGqWarps = 4, kGqThreads = kGqWarps * 32;
constexpr int kGqTile = kGqWarps * 16;    // rows per tile: 16 per warp
// dynamic shared memory of a kernel that streams rows of D bf16 with a ring of `stages` (K tile, V tile) pairs
__host__ __device__ constexpr int gq_tile_bytes(int D) { return kGqTile * D * 2; }           // 16 KB at D = 128
__host__ __device__ constexpr int gq_smem_bytes(int D, int stages) { return stages * 2 * gq_tile_bytes(D); }
constexpr int kGqMaxGroup = 16;
// Byte offset of 16-byte piece `piece` of row `row` in a shared-memory tile of D bf16 per row.
template <int D>
__device__ __forceinline__ uint32_t gq_tile_off(int row, int piece) {
  return D == 128 ? tile256_off(row, piece) : (uint32_t)(row * 128 + ((piece ^ (row & 7)) << 4));
}

// Per-warp triples in shared memory, laid over the tile ring once the rows have been consumed.
struct GqWarpTriples {
  float *o, *m, *l;     // [warps][16][D], [warps][16], [warps][16]
};

// One tile of K and of V (64 rows from r0; rows from r_end on are replaced by the last one before it) on its way to
// the ring stage at smem address `stage`.  A warp fetches the 16 rows that it will work on, so nothing but the warp
// has to wait for them.
template <int kGqD>
__device__ __forceinline__ void gq_load_tile(uint32_t stage, const uint8_t *Kg, const uint8_t *Vg, int r0, int r_end) {
  constexpr int kPieces = kGqD / 8;
#pragma unroll
  for (int x = 0; x < 16 * kPieces / 32; ++x) {
    const int idx = (threadIdx.x & 31) + x * 32, r = (threadIdx.x >> 5) * 16 + idx / kPieces, c = idx % kPieces;
    const size_t src = (size_t)min(r0 + r, r_end - 1) * (kGqD * 2) + c * 16;
    cp_async16(stage + gq_tile_off<kGqD>(r, c), Kg + src);
    cp_async16(stage + gq_tile_bytes(kGqD) + gq_tile_off<kGqD>(r, c), Vg + src);
  }
}

// The query vectors as the second operand of the scores: thread (g, t) of a warp holds head 8 n + g (head g % 4 where
// columns 4 .. 7 repeat the heads; zeros past G), 16 dims per step.  kMaxG: 1, 4, 8 or 16, at least G.
__host__ __device__ constexpr int gq_blocks(int max_g) { return (max_g + 7) / 8; }     // blocks of 8 columns
__host__ __device__ constexpr bool gq_repeats(int max_g) { return max_g <= 4; }        // columns 4 .. 7 repeat the heads of 0 .. 3
template <int kGqD, int kMaxG>
struct GqQuery { uint32_t b[gq_blocks(kMaxG)][kGqD / 16][2]; };
// q: G consecutive query vectors [G][D].  (To be asked for as early as may be: these loads cannot move ahead of
// asynchronous copies, or of a branch, by themselves.)
template <int kGqD, int kMaxG>
__device__ __forceinline__ GqQuery<kGqD, kMaxG> gq_load_query(const __nv_bfloat16 *q, int G) {
  const int g = (threadIdx.x & 31) >> 2, t = threadIdx.x & 3;
  GqQuery<kGqD, kMaxG> r;
#pragma unroll
  for (int n = 0; n < gq_blocks(kMaxG); ++n) {
    const int head = gq_repeats(kMaxG) ? g & 3 : 8 * n + g;
    const uint32_t *row = reinterpret_cast<const uint32_t *>(q + (size_t)head * kGqD);
#pragma unroll
    for (int ks = 0; ks < kGqD / 16; ++ks) {
      r.b[n][ks][0] = head < G ? row[ks * 8 + t] : 0u;
      r.b[n][ks][1] = head < G ? row[ks * 8 + 4 + t] : 0u;
    }
  }
  return r;
}

// Every thread of the CTA (kGqThreads of them) calls this with the same arguments.  The CTA's tiles are the 64
// rows from r_first + i * r_step for i = 0, 1, ... while that is below r_end (at least one).
// q: the G query vectors; Kg, Vg: first row of the slab.  Returns after a CTA barrier
// with the warps' triples in shared memory (gq_smem: gq_smem_bytes(D, kGqStages) of dynamic shared memory;
// kGqStages - 1 tiles are in flight while one is worked on).
template <int kGqD, int kGqStages, int kMaxG>
__device__ __forceinline__ GqWarpTriples gq_stream_rows(uint8_t *gq_smem, const GqQuery<kGqD, kMaxG> &q, int G,
                                                        const uint8_t *Kg, const uint8_t *Vg, int r_first, int r_step,
                                                        int r_end, float scale_log2) {
  static_assert(kGqD == 64 || kGqD == 128, "head_dim");
  constexpr int kGqTileBytes = gq_tile_bytes(kGqD);
  constexpr int kN = gq_blocks(kMaxG);
  constexpr bool kRepeat = gq_repeats(kMaxG); // for the low parts of the weights
  constexpr int kChains = 2;        // chains of MMAs that the scores of a block are summed in
  const int n_tiles = (r_end - r_first + r_step - 1) / r_step;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane >> 2, t = lane & 3;                                       // fragment row, column pair
  const uint32_t smem0 = (uint32_t)__cvta_generic_to_shared(gq_smem);
  auto load_tile = [&](int i) {                                                // tile i -> stage i % kGqStages
    gq_load_tile<kGqD>(smem0 + (i % kGqStages) * 2 * kGqTileBytes, Kg, Vg, r_first + i * r_step, r_end);
  };

#pragma unroll
  for (int i = 0; i < kGqStages - 1; ++i) {
    if (i < n_tiles) load_tile(i);
    cp_async_commit();
  }

  // o[n][j]: dims 16 j + g (and + 8) of heads 8 n + 2t, 2t + 1; m, l: those heads (l: this thread's keys)
  float o[kN][kGqD / 16][4], m[kN][2], l[kN][2];
#pragma unroll
  for (int n = 0; n < kN; ++n) {
#pragma unroll
    for (int j = 0; j < kGqD / 16; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[n][j][e] = 0.f;
    m[n][0] = m[n][1] = -INFINITY;
    l[n][0] = l[n][1] = 0.f;
  }

  for (int i = 0; i < n_tiles; ++i) {
    if (i + kGqStages - 1 < n_tiles) load_tile(i + kGqStages - 1);
    cp_async_commit();
    cp_async_wait<kGqStages - 1>();                             // tile i has landed (this thread's pieces)
    __syncwarp();                                               // ... and the warp's
    const uint32_t sk = smem0 + (i % kGqStages) * 2 * kGqTileBytes, sv = sk + kGqTileBytes;
    const int key0 = r_first + i * r_step + warp * 16;          // this warp's 16 rows of the tile

    if (key0 < r_end) {
      const bool ragged = key0 + 16 > r_end;
      const int mi = lane >> 3;
      // S^T = K Q^T: 16 keys x 8 heads per MMA
      float s[kN][kChains][4];
#pragma unroll
      for (int n = 0; n < kN; ++n)
#pragma unroll
        for (int c = 0; c < kChains; ++c)
#pragma unroll
          for (int e = 0; e < 4; ++e) s[n][c][e] = 0.f;
#pragma unroll
      for (int ks = 0; ks < kGqD / 16; ++ks) {
        uint32_t a[4];
        // matrices: (keys 0-7, dims lo), (keys 8-15, dims lo), (keys 0-7, dims hi), (keys 8-15, dims hi)
        ldmatrix_x4(a, sk + gq_tile_off<kGqD>(warp * 16 + (mi & 1) * 8 + (lane & 7), ks * 2 + (mi >> 1)));
#pragma unroll
        for (int n = 0; n < kN; ++n) mma_16816(s[n][ks % kChains], a, q.b[n][ks][0], q.b[n][ks][1]);
      }
      // Online softmax of heads 2t, 2t + 1: this thread holds keys g, g + 8.  The maximum moves only when a score
      // exceeds it by more than 2^8 (float32 sums and bf16 weights have the room).
      bool up = false;
#pragma unroll
      for (int n = 0; n < kN; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          float x = s[n][0][e];
#pragma unroll
          for (int c = 1; c < kChains; ++c) x += s[n][c][e];
          x *= scale_log2;
          if (ragged && key0 + g + 8 * (e >> 1) >= r_end) x = -INFINITY;
          s[n][0][e] = x;
          up = up || x > m[n][e & 1] + 8.f;
        }
      if (__any_sync(0xffffffffu, up)) {
#pragma unroll
        for (int n = 0; n < kN; ++n)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            float mx = fmaxf(s[n][0][e], s[n][0][e + 2]);
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
            const float m_new = fmaxf(m[n][e], mx);             // finite: key0 < r_end, so key 0 is valid
            const float alpha = exp2f(m[n][e] - m_new);         // m = -inf at first: 0
            m[n][e] = m_new;
            l[n][e] *= alpha;
#pragma unroll
            for (int j = 0; j < kGqD / 16; ++j) {
              o[n][j][e] *= alpha;
              o[n][j][e + 2] *= alpha;
            }
          }
      }
      constexpr int kParts = kRepeat ? 1 : 2;                   // operands that hold the weights
      uint32_t pb[kParts][kN][2];                               // P^T: keys 2t, 2t + 1 (| + 8) of head 8 n + g
#pragma unroll
      for (int n = 0; n < kN; ++n) {
        float p[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) p[e] = exp2f(s[n][0][e] - m[n][e & 1]);
        l[n][0] += p[0] + p[2];
        l[n][1] += p[1] + p[3];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const uint2 w = split2_bf16(p[2 * e], p[2 * e + 1]);
          if constexpr (kRepeat) {
            pb[0][n][e] = movmatrix_trans(t < 2 ? w.x : w.y);
          } else {
            pb[0][n][e] = movmatrix_trans(w.x);
            pb[kParts - 1][n][e] = movmatrix_trans(w.y);
          }
        }
      }
      // O^T += V^T P^T: 16 dims x 16 keys per ldmatrix
#pragma unroll
      for (int j = 0; j < kGqD / 16; ++j) {
        uint32_t a[4];
        // matrices: (dims lo, keys 0-7), (dims hi, keys 0-7), (dims lo, keys 8-15), (dims hi, keys 8-15)
        ldmatrix_x4_trans(a, sv + gq_tile_off<kGqD>(warp * 16 + (mi >> 1) * 8 + (lane & 7), j * 2 + (mi & 1)));
#pragma unroll
        for (int w = 0; w < kParts; ++w)
#pragma unroll
          for (int n = 0; n < kN; ++n) mma_16816(o[n][j], a, pb[w][n][0], pb[w][n][1]);
      }
    }
    __syncwarp();                                               // the warp's rows of the stage may be refilled
  }
  cp_async_wait<0>();
  __syncthreads();

  if constexpr (kRepeat) {                                      // high and low parts of the weights: columns 4 apart
#pragma unroll
    for (int j = 0; j < kGqD / 16; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[0][j][e] += __shfl_xor_sync(0xffffffffu, o[0][j][e], 2);
  }
  // merge the four warps' triples through shared memory (the tiles are no longer needed)
  float *sm_o = reinterpret_cast<float *>(gq_smem);             // [warps][16][D]
  float *sm_m = sm_o + kGqWarps * kGqMaxGroup * kGqD;           // [warps][16]
  float *sm_l = sm_m + kGqWarps * kGqMaxGroup;
#pragma unroll
  for (int n = 0; n < kN; ++n)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int head = 8 * n + 2 * t + e;
#pragma unroll
      for (int off = 4; off < 32; off <<= 1) l[n][e] += __shfl_xor_sync(0xffffffffu, l[n][e], off);
      if (head < G && (!kRepeat || t < 2)) {
        float *dst = sm_o + ((size_t)(warp * kGqMaxGroup + head)) * kGqD + g;
#pragma unroll
        for (int j = 0; j < kGqD / 16; ++j) {
          dst[16 * j] = o[n][j][e];
          dst[16 * j + 8] = o[n][j][e + 2];
        }
        if (g == 0) {
          sm_m[warp * kGqMaxGroup + head] = m[n][e];
          sm_l[warp * kGqMaxGroup + head] = l[n][e];
        }
      }
    }
  __syncthreads();
  return GqWarpTriples{sm_o, sm_m, sm_l};
}

// The CTA's triple for query h, output dimension d, from the warps' triples.
template <int kGqD>
__device__ __forceinline__ void gq_combine(const GqWarpTriples &w, int h, int d, float &acc, float &mc, float &lc) {
  mc = -INFINITY;
#pragma unroll
  for (int i = 0; i < kGqWarps; ++i) mc = fmaxf(mc, w.m[i * kGqMaxGroup + h]);
  acc = 0.f;
  lc = 0.f;
#pragma unroll
  for (int i = 0; i < kGqWarps; ++i) {
    const float mw = w.m[i * kGqMaxGroup + h];
    const float wgt = mw == -INFINITY ? 0.f : exp2f(mw - mc);
    acc = fmaf(wgt, w.o[((size_t)(i * kGqMaxGroup + h)) * kGqD + d], acc);
    lc = fmaf(wgt, w.l[i * kGqMaxGroup + h], lc);
  }
}

}  // namespace ag
