// MHA' of the Attention-Gate (Sec. 3.3) on the Blackwell tensor cores with
// float32-level accuracy.
//
// The gate's scores decide a hard threshold (Eq. 4), so bf16 rounding of Q', K',
// V' or of the attention weights would flip flags.  Every float32 operand x is
// therefore carried as a bf16 pair x = hi + lo (|x - hi - lo| <= 2^-17 |x|) and
// each product A B is evaluated as  Ahi Bhi + Ahi Blo + Alo Bhi  in the float32
// accumulator (the dropped lo*lo term is 2^-16 relative).  Gate heads of 64 take three parts (their sum is exactly
// x) and the six products down to 2^-16: with half the columns that costs about what two parts cost at 128.
//
// Structure as in the prefill kernel: warp 0 TMA, warp 1 tcgen05.mma issue,
// warps 2..5 softmax with one row per thread.  A query tile is 128 queries of
// one (sequence, gate head).  Scores are computed for pairs of key tiles (N = 128: an MMA of N = 64 waits for the 6 KB of
// operands it fetches, 52 cycles for 32 of arithmetic), weights and P V for tiles of 64 keys, whose V has two
// stages.  There is room for one pair's K only: it is taken in slices, each released as soon as its own MMAs have read it
// (a panel of 64 columns of both parts, or one part of 64-wide heads, the part with the fewest products
// first), so that the next pair's arrive while the rest of the scores and two P V run.
// Gate call, scores of one tile at a time | of pairs, us: 4 heads of 128, 333 tokens 31.0 | 31.0, 1500 50.1 | 48.6, 4096 102.3 |
// 95.7, 8192 265 | 247, 4 x 1999 155 | 149; 4 heads of 64, 4 x 1500 65.0 | 60.1, 8192 205 | 175.  A pair of 128-wide heads takes 3,072
// cycles of the tensor cores, which were busy 51 % of the time at 4096 tokens and are 60 %.  (The first tile's
// scores on their own, as a branch of the issuing warp: 8192 tokens of 64-wide heads 175 -> 213.)
//
// Work is the list of all (query tile, key tile) steps, query tiles in order
// and each one's key tiles in order.  The list is cut into equal segments, one
// CTA (one SM) each, so every SM gets the same number of steps whatever the
// shape of the causal triangle or the lengths of the sequences (a padded batch: the list holds the sequences' own
// tiles only; it is laid out on the device, from the lengths).  A segment crosses query tiles: the CTA handles
// its pieces one after the other, the loads of the next piece running under the
// tail of the current one.  Every piece leaves an un-normalised partial
// (O, m, l); gate_merge_out_kernel combines the pieces of a query tile and
// applies the gate's output layer and threshold.
//
// TMEM columns: scores of an even pair [0,128), of an odd one [128,256), O [256,256 + D) then 64 columns per part of P,
// each holding two tiles' weights (32 columns per tile).
#include "ag_common.cuh"
#include "mma_sync.cuh"
#include "umma.cuh"

namespace ag {

using namespace umma;

constexpr int kGaThreads = 192;
constexpr int kGaBM = 128, kGaBN = 64;
constexpr int kGaPanel = 128 * 128;                  // Q: [128 rows][64 bf16]
constexpr int kGaKvPanel = kGaBN * 128;              // K / V: [64 rows][64 bf16] = 8 KB
// Tiles of gate heads of width D (64 or 128): one or two 64-column panels.
template <int D>
struct GaCfg {
  static constexpr int kPanels = D / 64;
  static constexpr int kParts = D == 64 ? 3 : 2;          // bf16 parts per float32 value
  static constexpr int kProducts = kParts == 3 ? 6 : 3;   // products of parts (i, j), i + j < kParts
  static constexpr int kTile = kPanels * kGaPanel;        // one part of Q
  static constexpr int kKvTile = kPanels * kGaKvPanel;    // one part of K or V
  static constexpr int kKvStage = kParts * kKvTile;
  // K of a pair of key tiles: panels of [128 keys][64 columns], in slices
  static constexpr int kSlices = D == 64 ? kParts : kPanels;
  static constexpr int kSliceParts = D == 64 ? 1 : kParts;
  static constexpr int kSliceBytes = kSliceParts * kGaPanel;
  static_assert(kSlices * kSliceBytes == 2 * kKvStage, "K of a pair takes what two tiles of V do");
  static constexpr int kUsedBytes = kParts * kTile + 4 * kKvStage + 1024 + 256;   // Q + K of a pair + 2 V stages
  static constexpr uint32_t kColO = 256, kColP = kColO + D;
  static_assert(kColP + 64 * kParts <= 512, "tensor memory");
  // parts of the first and of the second operand of product t
  __host__ __device__ static constexpr int first(int t) { return t == 0 || t == 1 || t == 3 ? 0 : (t == 2 || t == 5 ? 1 : 2); }
  __host__ __device__ static constexpr int second(int t) { return t == 0 || t == 2 || t == 4 ? 0 : (t == 1 || t == 5 ? 1 : 2); }
  // one CTA per SM whatever D (each takes all of tensor memory: a second one on the SM would wait for the first
  // to end while other SMs stand idle)
  static constexpr int kSmemBytes = kUsedBytes > 120 * 1024 ? kUsedBytes : 120 * 1024;
};
constexpr uint32_t kGaColS = 0, kGaTmemCols = 512;
constexpr float kGaRescaleThreshold = 8.f;

constexpr int kGaMaxSeg = 256;       // segments at most (one per SM)
constexpr int kGaOverhead = 2;       // set-up + epilogue of a query tile, in key tiles (even)

// The list of work: for every sequence b, gate head g and query tile q of the sequence's own length, kGaOverhead places
// that stand for the tile's set-up and epilogue and one place per key tile.  The list is cut into n_seg segments
// of equal length; the key tiles of a query tile inside a segment are a piece.  All lengths are even, so a piece
// starts on a 128-key boundary and its first tile holds a key every row of the query tile may see.
struct GateAttnArgs {
  const int32_t *seq_lens;  // [B] or NULL: tokens past seq_lens[b] are padding
  float *part_o;            // [items, 128, D] un-normalised partial outputs
  float *part_ml;           // [items, 128, 2]   running max (log2 units) and sum per row
  int n, n_qtiles, batch, gate_heads, GD, causal;
  int n_seg;                // segments (= CTAs of the attention kernel)
  float scale_log2;
};

// One map per part (all 3 encoded): boxes of a query tile's rows and of a key tile's.
struct GateAttnMaps { CUtensorMap q[3], kv[3]; };

// Key tiles (64 keys) of query tile q (128 queries) of a sequence of nq query tiles, and list places: of the tile,
// before the tile within its (sequence, gate head), and of a whole (sequence, gate head).
__host__ __device__ inline int ga_key_tiles(int q, int nq, int causal) { return 2 * (causal ? q + 1 : nq); }
__host__ __device__ inline int ga_tile_places(int q, int nq, int causal) { return ga_key_tiles(q, nq, causal) + kGaOverhead; }
__host__ __device__ inline int ga_places_before(int q, int nq, int causal) {
  return causal ? q * (q + 1) + kGaOverhead * q : q * (2 * nq + kGaOverhead);
}
__host__ __device__ inline int ga_head_places(int nq, int causal) { return ga_places_before(nq, nq, causal); }
__device__ inline int ga_seq_tiles(const GateAttnArgs &a, int b) {
  return a.seq_lens == nullptr ? a.n_qtiles : (min(max(a.seq_lens[b], 0), a.n) + kGaBM - 1) / kGaBM;
}
__device__ inline int ga_seg_len(const GateAttnArgs &a, int total) {
  return max(2, ((total + a.n_seg - 1) / a.n_seg + 1) & ~1);
}
// Whole-warp call: places of the list in all, and before sequence b_end.
__device__ inline int ga_total(const GateAttnArgs &a, int b_end, int &before) {
  if (a.seq_lens == nullptr) {
    const int per = a.gate_heads * ga_head_places(a.n_qtiles, a.causal);
    before = b_end * per;
    return a.batch * per;
  }
  int total = 0, bef = 0;
  for (int b = threadIdx.x & 31; b < a.batch; b += 32) {
    const int v = a.gate_heads * ga_head_places(ga_seq_tiles(a, b), a.causal);
    total += v;
    if (b < b_end) bef += v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    total += __shfl_xor_sync(0xffffffffu, total, o);
    bef += __shfl_xor_sync(0xffffffffu, bef, o);
  }
  before = bef;
  return total;
}

// Where a CTA stands in the list: sequence, gate head, query tile of nq, place within the tile, places left.
struct GaWalk { int b, g, q, nq, v, left; };
struct GaPiece { int b, g, qt, kv_begin, n_kv; };
// Whole-warp call: the start of segment seg.
__device__ inline GaWalk ga_start(const GateAttnArgs &a, int seg) {
  GaWalk w = {};
  int before;
  const int total = ga_total(a, 0, before), len = ga_seg_len(a, total);
  int x = seg * len;
  w.left = min(len, total - x);
  if (w.left <= 0) return w;
  if (a.seq_lens == nullptr) {
    const int per = a.gate_heads * ga_head_places(a.n_qtiles, a.causal);
    w.b = x / per;
    x -= w.b * per;
  } else {
    const int lane = threadIdx.x & 31;
    for (int b0 = 0;; b0 += 32) {                    // (x < total: some sequence holds it)
      const int v = b0 + lane < a.batch ? a.gate_heads * ga_head_places(ga_seq_tiles(a, b0 + lane), a.causal) : 0;
      int incl = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int up = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += up;
      }
      const unsigned past = __ballot_sync(0xffffffffu, incl > x);
      if (past != 0) {
        const int l = __ffs(past) - 1;
        w.b = b0 + l;
        x -= __shfl_sync(0xffffffffu, incl - v, l);
        break;
      }
      x -= __shfl_sync(0xffffffffu, incl, 31);
      if (b0 + 32 >= a.batch) { w.left = 0; return w; }
    }
  }
  w.nq = ga_seq_tiles(a, w.b);
  const int head = ga_head_places(w.nq, a.causal);
  w.g = x / head;
  const int y = x - w.g * head;
  if (a.causal) {
    int q = (int)((sqrtf(4.f * (float)y + 9.f) - 3.f) * 0.5f);      // q (q + 1) + 2 q = y
    while (q > 0 && ga_places_before(q, w.nq, 1) > y) --q;
    while (ga_places_before(q + 1, w.nq, 1) <= y) ++q;
    w.q = q;
  } else {
    w.q = y / ga_tile_places(0, w.nq, 0);
  }
  w.v = y - ga_places_before(w.q, w.nq, a.causal);
  return w;
}
// The next piece of the segment; false at its end.
__device__ inline bool ga_next(const GateAttnArgs &a, GaWalk &w, GaPiece &p) {
  while (w.left > 0) {
    const int tile = ga_tile_places(w.q, w.nq, a.causal), end = min(tile, w.v + w.left);
    const int k0 = max(w.v - kGaOverhead, 0);
    p.b = w.b; p.g = w.g; p.qt = w.q;
    p.kv_begin = k0;
    p.n_kv = end - kGaOverhead - k0;
    w.left -= end - w.v;
    w.v = end;
    if (end == tile) {
      w.v = 0;
      if (++w.q == w.nq) {
        w.q = 0;
        if (++w.g == a.gate_heads) {
          w.g = 0;
          do {
            ++w.b;
            w.nq = w.b < a.batch ? ga_seq_tiles(a, w.b) : 0;
          } while (w.nq == 0 && w.b < a.batch);
          if (w.nq == 0) w.left = 0;
        }
      }
    }
    if (p.n_kv > 0) return true;
  }
  return false;
}
// Partial slot of the piece of query tile (prob, qt) that lies in segment seg: consecutive pieces
// differ in the query tile, the segment or both, so the sum is unique and grows along the list.
__host__ __device__ inline int ga_slot(int prob, int qt, int n_qtiles, int seg) {
  return prob * n_qtiles + qt + seg;
}

template <int kGaD>
__global__ void __launch_bounds__(kGaThreads, 1)
gate_attn_tc_kernel(const __grid_constant__ GateAttnMaps tm, const __grid_constant__ GateAttnArgs a) {
  using C = GaCfg<kGaD>;
  constexpr int kGaTile = C::kTile, kGaKvTile = C::kKvTile, kGaKvStage = C::kKvStage;
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *sQ = smem;                    // [part]
  // [slice][part of the slice][128 keys][64 columns]; of 64-wide heads slice s holds part kParts - 1 - s
  uint8_t *sK = sQ + C::kParts * kGaTile;
  uint8_t *sV = sK + 2 * kGaKvStage;
  uint64_t *bars = reinterpret_cast<uint64_t *>(sV + 2 * kGaKvStage);
  uint64_t *q_empty = bars, *o_free = bars + 1;
  uint64_t *k_full = bars + 2, *k_empty = bars + 5;                          // [slice]
  uint64_t *v_full = bars + 8, *v_empty = bars + 10, *s_full = bars + 12;    // [2]
  // p_ready[2], pv_done[2]: even / odd tiles.  P is double-buffered (32 of each half's 64 columns per tile), so
  // the weights of tile t are written while the P V of tile t - 1 runs; a softmax warp may be a tile ahead
  // of a slower one, never two (the weights of tile t + 2 wait for the P V of tile t).
  uint64_t *p_ready = bars + 14, *pv_done = bars + 16;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(bars + 18);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Every role walks the pieces of this CTA's segment with the same arithmetic;
  // tiles are numbered t = 0, 1, ... across the pieces (stage of V, P and the P V barrier t & 1, in their use
  // number t >> 1), pairs of tiles u = t >> 1 (K slices in their use number u, scores u & 1 in their use
  // number u >> 1), pieces pc = 0, 1, ...

  if (threadIdx.x == 0) {
    for (int s = 0; s < 2; ++s) {
      mbar_init(&v_full[s], 1); mbar_init(&v_empty[s], 1);
      mbar_init(&s_full[s], 1);
    }
    for (int s = 0; s < C::kSlices; ++s) { mbar_init(&k_full[s], 1); mbar_init(&k_empty[s], 1); }
    mbar_init(&p_ready[0], 128); mbar_init(&p_ready[1], 128);
    mbar_init(&pv_done[0], 1); mbar_init(&pv_done[1], 1);
    mbar_init(q_empty, 1);
    mbar_init(o_free, 128);
    fence_barrier_init();
#pragma unroll
    for (int i = 0; i < C::kParts; ++i) { prefetch_tensormap(&tm.q[i]); prefetch_tensormap(&tm.kv[i]); }
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, kGaTmemCols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();                                        // the projections are there
  pdl_launch_dependents();
  GaWalk walk = ga_start(a, (int)blockIdx.x);
  GaPiece pz = {};

  if (warp == 0) {
    if (lane == 0) {
      int t = 0;
      // Pair i of the piece, pair u of the segment; columns of [Q' | K' | V']: g D, GD + g D, 2 GD + g D.  With the first pair
      // of a piece comes its Q, in slices of the same shape: slice s of the scores needs no more of Q than slices 0 .. s.
      auto load_k = [&](int u, int i, int pc) -> bool {
        const int y = (pz.kv_begin + 2 * i) * kGaBN;
        if (i == 0 && !mbar_wait(q_empty, (pc & 1) ^ 1)) return false;      // the previous piece's last Q K^T has read Q
#pragma unroll
        for (int s = 0; s < C::kSlices; ++s) {
          if (!mbar_wait(&k_empty[s], (u & 1) ^ 1)) return false;
          mbar_arrive_expect_tx(&k_full[s], i == 0 ? 2 * C::kSliceBytes : C::kSliceBytes);
          const int col = pz.g * kGaD + (kGaD == 64 ? 0 : s * 64);
#pragma unroll
          for (int x = 0; x < C::kSliceParts; ++x) {
            if (i == 0)
              tma_load_3d(kGaD == 64 ? sQ + s * kGaTile : sQ + x * kGaTile + s * kGaPanel, &tm.q[kGaD == 64 ? s : x], &k_full[s], col,
                          pz.qt * kGaBM, pz.b);
#pragma unroll
            for (int r = 0; r < 2; ++r)
              tma_load_3d(sK + s * C::kSliceBytes + x * kGaPanel + r * kGaKvPanel, &tm.kv[kGaD == 64 ? C::kParts - 1 - s : x],
                          &k_full[s], a.GD + col, y + r * kGaBN, pz.b);
          }
        }
        return true;
      };
      auto load_v = [&](int t, int b, int x, int y) -> bool {
        const int st = t & 1;
        if (!mbar_wait(&v_empty[st], ((t >> 1) & 1) ^ 1)) return false;
        mbar_arrive_expect_tx(&v_full[st], kGaKvStage);
#pragma unroll
        for (int i = 0; i < C::kParts; ++i)
#pragma unroll
          for (int p = 0; p < C::kPanels; ++p)
            tma_load_3d(sV + st * kGaKvStage + i * kGaKvTile + p * kGaKvPanel, &tm.kv[i], &v_full[st], x + p * 64, y, b);
        return true;
      };
      // in the order in which the buffers become free: K of pair u + 1 (with Q where a piece begins), then the V tiles of pair u
      // (those of the first pair at once)
      bool more = ga_next(a, walk, pz), ok = more && load_k(0, 0, 0);
      for (int pc = 1; ok && more; ++pc) {
        const int pairs = pz.n_kv / 2, b = pz.b, xv = 2 * a.GD + pz.g * kGaD, kv_begin = pz.kv_begin;
        for (int i = 0; i < pairs && ok; ++i, t += 2) {
          const int y = (kv_begin + 2 * i) * kGaBN;
          if (t == 0) ok = load_v(0, b, xv, y) && load_v(1, b, xv, y + kGaBN);
          if (i + 1 < pairs) ok = ok && load_k((t >> 1) + 1, i + 1, pc);
          else if ((more = ga_next(a, walk, pz))) ok = ok && load_k((t >> 1) + 1, 0, pc);
          if (t != 0) ok = ok && load_v(t, b, xv, y) && load_v(t + 1, b, xv, y + kGaBN);
        }
      }
    }
  } else if (warp == 1) {
    // every lane runs the control flow (operands stay warp-uniform); one elected lane issues
    constexpr uint32_t idesc_qk = idesc_bf16_f32(kGaBM, 2 * kGaBN, false, false);
    constexpr uint32_t idesc_pv = idesc_bf16_f32(kGaBM, kGaD, false, true);
    const uint64_t dq = desc_kmajor_sw128(smem_u32(sQ)), dk = desc_kmajor_sw128(smem_u32(sK));
    const uint64_t dv = desc_mnmajor_sw128(smem_u32(sV), kGaKvPanel);
    const uint32_t q_lo = (uint32_t)dq, q_hi = (uint32_t)(dq >> 32);
    const uint32_t k_lo = (uint32_t)dk, k_hi = (uint32_t)(dk >> 32);
    const uint32_t v_lo = (uint32_t)dv, v_hi = (uint32_t)(dv >> 32);
    auto issue_qk = [&](int u, bool last) -> bool {   // u: pair number across the pieces
      const uint32_t d = tmem + kGaColS + (u & 1) * 128;
#pragma unroll
      for (int s = 0; s < C::kSlices; ++s) {
        if (!mbar_wait(&k_full[s], u & 1)) return false;
        tc_fence_after_sync();
        if (elect_one()) {
#pragma unroll
          for (int t = 0; t < C::kProducts; ++t) {
            if (kGaD == 64 && C::second(t) != C::kParts - 1 - s) continue;
            const uint32_t qa = q_lo + ((C::first(t) * kGaTile + (kGaD == 64 ? 0 : s * kGaPanel)) >> 4);
            const uint32_t ka = k_lo + ((s * C::kSliceBytes + (kGaD == 64 ? 0 : C::second(t) * kGaPanel)) >> 4);
#pragma unroll
            for (int k = 0; k < 4; ++k)               // a panel is 64 columns
              mma_ss_lohi(d, qa + ((k * 32) >> 4), q_hi, ka + ((k * 32) >> 4), k_hi, idesc_qk,
                          s != 0 || k != 0 || (kGaD != 64 && t != 0));
          }
          mma_commit(&k_empty[s]);
          if (s + 1 == C::kSlices) {
            mma_commit(&s_full[u & 1]);
            if (last) mma_commit(q_empty);            // Q may be replaced by the next piece's
          }
        }
        __syncwarp();
      }
      return true;
    };
    auto issue_pv = [&](int t, bool first) -> bool {  // first: of its piece
      const int st = t & 1;
      if (!mbar_wait(&p_ready[st], (t >> 1) & 1)) return false;
      if (!mbar_wait(&v_full[st], (t >> 1) & 1)) return false;
      tc_fence_after_sync();
      const uint32_t vb = v_lo + ((st * kGaKvStage) >> 4);
      if (elect_one()) {
#pragma unroll
        for (int t = 0; t < C::kProducts; ++t) {
          const uint32_t pa = tmem + C::kColP + C::first(t) * 64 + st * (kGaBN / 2);
          const uint32_t va = vb + ((C::second(t) * kGaKvTile) >> 4);
#pragma unroll
          for (int k = 0; k < kGaBN / 16; ++k)
            mma_ts_lohi(tmem + C::kColO, pa + k * 8, va + ((k * 2048) >> 4), v_hi, idesc_pv, !first || (t | k) != 0);
        }
        mma_commit(&v_empty[st]);
        mma_commit(&pv_done[st]);
      }
      __syncwarp();
      return true;
    };
    // The scores of a pair ahead of the two P V of the pair before; those of a piece's first pair behind the piece before
    // (between its last two P V, its Q is awaited too early: 4096 tokens 99.3 us against 96.6).  One place in the code for
    // each: the loops stay small beside the softmax warps' code.
    bool ok = true;
    int u0 = 0;                                      // number of the piece's first pair
    for (int pc = 0; ok && ga_next(a, walk, pz); ++pc) {
      const int pairs = pz.n_kv / 2;
#pragma unroll 1
      for (int i = -1; i < pairs && ok; ++i) {
        if (i + 1 < pairs) ok = issue_qk(u0 + i + 1, i + 2 == pairs);
        if (i < 0) continue;
        // the first P V of a piece overwrites O: the previous piece's epilogue must have read it
        if (i == 0 && pc > 0) ok = ok && mbar_wait(o_free, (pc - 1) & 1);
#pragma unroll 1
        for (int h = 0; h < 2; ++h) ok = ok && issue_pv(2 * (u0 + i) + h, i == 0 && h == 0);
      }
      u0 += pairs;
    }
  } else {
    const int quad = warp & 3;
    const int row = quad * 32 + lane;
    const uint32_t tm_lane = tmem + ((uint32_t)(quad * 32) << 16);
    bool ok = true;
    int t0 = 0;                                      // tile number of the piece's first tile

    while (ok && ga_next(a, walk, pz)) {
    const int n_kv = pz.n_kv, kv_begin = pz.kv_begin;
    const int j = pz.qt * kGaBM + row;
    const bool valid = j < a.n;
    const int jc = min(j, a.n - 1);
    // keys below bound are visible (bidirectional: the sequence's own tokens, not its padding)
    const int seq_len = a.seq_lens ? a.seq_lens[pz.b] : a.n;
    const int bound = a.causal ? jc + 1 : seq_len;
    float m = -INFINITY, l = 0.f;
    for (int i = 0; i < n_kv && ok; ++i) {
      const int t = t0 + i;
      ok = mbar_wait(&s_full[(t >> 1) & 1], (t >> 2) & 1);
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t tS = tm_lane + kGaColS + ((t >> 1) & 1) * 128 + (t & 1) * kGaBN;
      const int nvalid = min(max(bound - (kv_begin + i) * kGaBN, 0), kGaBN);
      const bool full = nvalid >= kGaBN;

      uint32_t r[kGaBN];
      tmem_ld_x64_sync(tS, r);
      if (!full) {
#pragma unroll
        for (int e = 0; e < kGaBN; ++e)
          if (e >= nvalid) r[e] = 0xff800000u;        // -inf: weight 0 below
      }
      // eight independent chains, two elements per instruction
      float mx[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) mx[q] = max3_f32(__uint_as_float(r[q]), __uint_as_float(r[q + 8]), __uint_as_float(r[q + 16]));
#pragma unroll
      for (int e = 24; e + 8 < kGaBN; e += 16)
#pragma unroll
        for (int q = 0; q < 8; ++q) mx[q] = max3_f32(mx[q], __uint_as_float(r[e + q]), __uint_as_float(r[e + q + 8]));
#pragma unroll
      for (int q = 0; q < 8; ++q) mx[q] = fmaxf(mx[q], __uint_as_float(r[kGaBN - 8 + q]));
      float tmax = max3_f32(max3_f32(mx[0], mx[1], mx[2]), max3_f32(mx[3], mx[4], mx[5]), fmaxf(mx[6], mx[7]));
      tmax *= a.scale_log2;
      // The first tile of a piece holds a key visible to every row (key 0, or a tile wholly before
      // the query tile; the list has no tiles of padding).  m = -inf after it takes scores of -inf, out of
      // inputs that overflow: every weight is 0 then.
      float m_new;
      if (i == 0) m_new = tmax;
      else m_new = (tmax > m + kGaRescaleThreshold) ? tmax : m;
      const bool rescale = (i > 0) && __any_sync(0xffffffffu, m_new != m);
      const float alpha = (i == 0 || m == -INFINITY) ? 0.f : fast_exp2(m - m_new);
      l *= alpha;
      const float m_exp = m_new == -INFINITY ? 0.f : m_new;    // exponent offset: keeps -inf - (-inf) out

      // Only a rescale of O has to wait for the P V of tile t - 1 (the next phase of that barrier is the P V of
      // tile t + 1, which cannot have been issued yet: the parity is unambiguous)
      if (rescale) {
        ok = mbar_wait(&pv_done[(t - 1) & 1], ((t - 1) >> 1) & 1);
        if (!ok) break;
        tc_fence_after_sync();
#pragma unroll 1
        for (int c = 0; c < kGaD / 32; ++c) {
          uint32_t r[32];
          tmem_ld_x32_sync(tm_lane + C::kColO + c * 32, r);
#pragma unroll
          for (int e = 0; e < 32; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * alpha);
          tmem_st_x32(tm_lane + C::kColO + c * 32, r);
        }
      }
      // this tile's P buffer was last read by the P V of tile t - 2
      if (t >= 2) {
        ok = mbar_wait(&pv_done[t & 1], ((t >> 1) & 1) ^ 1);
        if (!ok) break;
        tc_fence_after_sync();
      }

      float rs[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c = 0; c < kGaBN / 16; ++c) {
        uint32_t pk[C::kParts][8];
#pragma unroll
        for (int e = 0; e < 16; e += 2) {
          float x0, x1;
          fma_f32x2(x0, x1, __uint_as_float(r[c * 16 + e]), __uint_as_float(r[c * 16 + e + 1]), a.scale_log2,
                    a.scale_log2, -m_exp, -m_exp);
          float p0 = fast_exp2(x0), p1 = fast_exp2(x1);
          const int k = ((e >> 1) & 3) * 2;
          add_f32x2(rs[k], rs[k + 1], rs[k], rs[k + 1], p0, p1);
#pragma unroll
          for (int i = 0; i + 1 < C::kParts; ++i) pk[i][e >> 1] = take_bf16x2(p0, p1);
          pk[C::kParts - 1][e >> 1] = pack_bf16x2(p0, p1);
        }
#pragma unroll
        for (int i = 0; i < C::kParts; ++i)
          tmem_st_x8(tm_lane + C::kColP + i * 64 + (t & 1) * (kGaBN / 2) + c * 8, pk[i]);
      }
      l += ((rs[0] + rs[1]) + (rs[2] + rs[3])) + ((rs[4] + rs[5]) + (rs[6] + rs[7]));
      m = m_new;
      tmem_st_wait();
      tc_fence_before_sync();
      mbar_arrive(&p_ready[t & 1]);
    }

    if (ok) {
      ok = mbar_wait(&pv_done[(t0 + n_kv - 1) & 1], ((t0 + n_kv - 1) >> 1) & 1);
      tc_fence_after_sync();
    }
    if (ok) {
      const size_t it = (size_t)ga_slot(pz.b * a.gate_heads + pz.g, pz.qt, a.n_qtiles, (int)blockIdx.x);
      float *op = a.part_o + (it * kGaBM + row) * kGaD;
#pragma unroll 1
      for (int c = 0; c < kGaD / 32; ++c) {
        uint32_t r[32];
        tmem_ld_x32_sync(tm_lane + C::kColO + c * 32, r);
        if (c + 1 == kGaD / 32) {                                // O is in registers: the next piece may overwrite it
          tc_fence_before_sync();
          mbar_arrive(o_free);
        }
        if (valid) {
#pragma unroll
          for (int e = 0; e < 32; e += 4)
            *reinterpret_cast<uint4 *>(op + c * 32 + e) = make_uint4(r[e], r[e + 1], r[e + 2], r[e + 3]);
        }
      }
      if (valid) *reinterpret_cast<float2 *>(a.part_ml + (it * kGaBM + row) * 2) = make_float2(m, l);
    }
    t0 += n_kv;
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, kGaTmemCols);
}

// The split-K merge of MHA' and the gate's output layer in one pass (Eq. 3, Eq. 4):
//   H'[t, g * D + c] = sum_s w_s O_s[r, c] / sum_s w_s l_s,  w_s = 2^(m_s - max_s m_s)
//   s[t, i] = H'[t, :] Wo_g[:, i];  flag = s + gamma_i > logit(tau)
// One CTA = kTok tokens (16, or 8 or 4 where the tokens would not fill the SMs), 16 / kTok warps per token.  A warp
// merges the token's row of its share of the gate heads (a lane per D / 32 columns: every access is one whole row), eight
// pieces' rows in flight at a time under a running maximum, into shared memory; then the warps share the
// reduction, 16 columns of H' at a time, as m16n8k16 MMAs of the 16 tokens against 32 heads of Wo.
// Every float32 of H' enters as three bf16 (8 + 8 + 8 mantissa bits: exactly its value), so nothing of it
// is lost, and Wo is bf16 as it comes.  The warps' sums are added in a fixed order.  H' never goes to global
// memory.  (With the products on CUDA cores, operands from shared memory, this was 18 us at 4,096 tokens
// and 141 us at 8 x 4,096.)  Wo is fetched before the wait for MHA', which it does not depend on.  Bound by latency: one trip to
// L2 per eight pieces (the maxima used to be a trip of their own, two pieces at a time) and few tokens spread over all
// SMs: pass of 333 tokens 123 -> 118 us, of 1,000 tokens 83 -> 75, of 4 x 1,500 (64-wide heads) 123 -> 119.
constexpr int kMoWarps = 16, kMoThreads = kMoWarps * 32;
template <int N> struct FloatVec;
template <> struct FloatVec<2> { using type = float2; };
template <> struct FloatVec<4> { using type = float4; };
constexpr int kMoRedPitch = 33;                                  // floats per token of a warp's sums (32 heads)
constexpr int kMoRedBytes = kMoWarps * 16 * kMoRedPitch * 4;
__host__ __device__ constexpr int mo_w_bytes(int GD) { return GD * 64 > kMoRedBytes ? GD * 64 : kMoRedBytes; }
__host__ __device__ constexpr int mo_smem_bytes(int GD) { return mo_w_bytes(GD) + 16 * (GD + 8) * 4; }
constexpr int kMoPieceBytes = 2 * kMoThreads * 4;                // static: where the pieces of each gate head lie
constexpr int kMaxSmemBytes = 227 * 1024;                        // of one CTA
// Byte offset of 16-byte piece `piece` (8 heads) of row `c` of the staged slice of Wo: 64-byte rows, pieces XOR-ed so
// that the eight rows one ldmatrix reads fall into different banks.
__device__ __forceinline__ uint32_t mo_w_off(int c, int piece) { return (uint32_t)(c * 64 + ((piece ^ ((c >> 1) & 3)) << 4)); }

template <int kGaD, int kTok>
__global__ void __launch_bounds__(kMoThreads)
gate_merge_out_kernel(const __grid_constant__ GateAttnArgs a, const __nv_bfloat16 *__restrict__ Wo,
                      const float *__restrict__ gamma, float logit_tau, int h, float *__restrict__ scores,
                      uint8_t *__restrict__ flags) {
  extern __shared__ __align__(16) unsigned char mo_smem[];
  unsigned char *Ws = mo_smem;                                   // [GD][32] bf16, then the warps' sums
  float *red = reinterpret_cast<float *>(mo_smem);               // [warps][16 tokens][33]
  float *Hs = reinterpret_cast<float *>(mo_smem + mo_w_bytes(a.GD));     // [16][GD + 8]
  const int pitch = a.GD + 8;
  __shared__ int seg_first[2][kMoThreads];           // per gate head: first segment, number of pieces
  static_assert(sizeof(seg_first) == kMoPieceBytes, "gate_attn_tc_supported");
  const int tiles_per_seq = (a.n + kTok - 1) / kTok;
  const int b = blockIdx.x / tiles_per_seq, t0 = (blockIdx.x % tiles_per_seq) * kTok;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = t0 + warp % kTok;
  float *hrow = Hs + (warp % kTok) * pitch;
  // heads i0 .. i0 + 31 of Wo
  auto stage_wo = [&](int i0) {
    const uint32_t ws = smem_u32(Ws);
    for (int x = threadIdx.x; x < a.GD * 4; x += kMoThreads) {
      const int c = x >> 2, i = i0 + (x & 3) * 8;
      const uint32_t off = mo_w_off(c, x & 3);
      if ((h & 7) == 0 && i < h) {
        cp_async16(ws + off, Wo + (size_t)c * h + i);
      } else {
        __nv_bfloat16 *dst = reinterpret_cast<__nv_bfloat16 *>(Ws + off);
#pragma unroll
        for (int e = 0; e < 8; ++e) dst[e] = i + e < h ? Wo[(size_t)c * h + i + e] : __float2bfloat16_rn(0.f);
      }
    }
    cp_async_commit();
  };
  // The CTA's tokens lie in one query tile: which segments hold its pieces is looked up once per gate head.
  auto find_pieces = [&] {
    const int qt = t0 / kGaBM, nq = ga_seq_tiles(a, b);
    int before;
    const int len = ga_seg_len(a, ga_total(a, b, before));
    for (int g = lane; g < a.gate_heads; g += 32) {
      // the query tile's key tiles [x0, x1) of the list lie in consecutive segments, one piece in each
      const int x0 = before + g * ga_head_places(nq, a.causal) + ga_places_before(qt, nq, a.causal) + kGaOverhead;
      const int x1 = x0 + ga_key_tiles(qt, nq, a.causal);
      seg_first[0][g] = x0 / len;
      seg_first[1][g] = (x1 - 1) / len - x0 / len + 1;
    }
  };
  stage_wo(0);
  // What does not depend on MHA' is done before the wait for it (MHA' lets this kernel start once it has itself waited
  // for all that came before: inputs of the call are there).
  const bool padding_only = a.seq_lens != nullptr && t0 >= a.seq_lens[b];
  if (warp == 0 && !padding_only) find_pieces();
  const float gamma0 = gamma && threadIdx.x / kTok < min(h, 32) ? gamma[threadIdx.x / kTok] : 0.f;
  pdl_wait();                                        // (no early trigger of the next kernel: 2 % of the pass lost with it)
  if (padding_only) {
    // flags 0, scores left as they are
    cp_async_wait<0>();
    const int tok = threadIdx.x % kTok;
    for (int i = threadIdx.x / kTok; i < h; i += kMoThreads / kTok)
      if (t0 + tok < a.n) flags[((size_t)b * h + i) * a.n + t0 + tok] = 0;
    return;
  }
  __syncthreads();
  if (t < a.n) {
    constexpr int kU = kTok / 4, kP = 8 / kU;        // gate heads, and pieces of each, in flight together
    const int qt = t / kGaBM, r = t % kGaBM;
    for (int g0 = (warp / kTok) * kU; g0 < a.gate_heads; g0 += 4) {
      constexpr int kV = kGaD / 32;                  // columns per lane
      using Vec = typename FloatVec<kV>::type;
      size_t row0[kU];
      int ns[kU], ns_max = 0;
      float acc[kU][kV], lsum[kU], m[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const int g = min(g0 + u, a.gate_heads - 1), prob = b * a.gate_heads + g;
        ns[u] = seg_first[1][g];
        row0[u] = (size_t)ga_slot(prob, qt, a.n_qtiles, seg_first[0][g]) * kGaBM + r;   // + s * 128 per piece
        ns_max = max(ns_max, ns[u]);
        m[u] = -INFINITY;
        lsum[u] = 0.f;
#pragma unroll
        for (int e = 0; e < kV; ++e) acc[u][e] = 0.f;
      }
      for (int s0 = 0; s0 < ns_max; s0 += kP) {
        float2 ml[kU][kP];
        Vec o4[kU][kP];
#pragma unroll
        for (int u = 0; u < kU; ++u)
#pragma unroll
          for (int p = 0; p < kP; ++p) {
            // (past the last piece: the last one again, at weight 0)
            const size_t row = row0[u] + (size_t)min(s0 + p, ns[u] - 1) * kGaBM;
            ml[u][p] = *reinterpret_cast<const float2 *>(a.part_ml + row * 2);
            o4[u][p] = *reinterpret_cast<const Vec *>(a.part_o + row * kGaD + lane * kV);
          }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          float m_new = m[u];
#pragma unroll
          for (int p = 0; p < kP; ++p) m_new = fmaxf(m_new, ml[u][p].x);
          const float alpha = fast_exp2(m[u] - m_new);         // m = -inf at first: 0
          m[u] = m_new;
          lsum[u] *= alpha;
#pragma unroll
          for (int e = 0; e < kV; ++e) acc[u][e] *= alpha;
#pragma unroll
          for (int p = 0; p < kP; ++p) {
            const float w = s0 + p < ns[u] ? fast_exp2(ml[u][p].x - m_new) : 0.f;
            const float *o = reinterpret_cast<const float *>(&o4[u][p]);
#pragma unroll
            for (int e = 0; e < kV; ++e) acc[u][e] = fmaf(w, o[e], acc[u][e]);
            lsum[u] = fmaf(w, ml[u][p].y, lsum[u]);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        if (g0 + u < a.gate_heads) {
          const float inv = 1.f / lsum[u];
          Vec hv;
#pragma unroll
          for (int e = 0; e < kV; ++e) reinterpret_cast<float *>(&hv)[e] = acc[u][e] * inv;
          *reinterpret_cast<Vec *>(hrow + (g0 + u) * kGaD + lane * kV) = hv;
        }
      }
    }
  }
  // (rows of H' without a token hold anything: a row of an MMA's first operand reaches its own row of the result only)
  const int g = lane >> 2, tq = lane & 3, mi = lane >> 3;
  for (int i0 = 0; i0 < h; i0 += 32) {
    if (i0 > 0) {
      __syncthreads();                               // the previous round's sums have been read
      stage_wo(i0);
    }
    cp_async_wait<0>();
    __syncthreads();                                 // H' rows and this slice of Wo are complete
    float c[4][4];                                   // 16 tokens x 32 heads, this warp's share of the reduction
#pragma unroll
    for (int nb = 0; nb < 4; ++nb)
#pragma unroll
      for (int e = 0; e < 4; ++e) c[nb][e] = 0.f;
    const uint32_t ws = smem_u32(Ws);
    for (int k0 = warp * 16; k0 < a.GD; k0 += kMoWarps * 16) {
      uint32_t ah[3][4];                             // the three bf16 parts of the fragment of H'
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        float2 x = *reinterpret_cast<const float2 *>(Hs + (g + (f & 1) * 8) * pitch + k0 + (f >> 1) * 8 + 2 * tq);
        ah[0][f] = take_bf16x2(x.x, x.y);
        ah[1][f] = take_bf16x2(x.x, x.y);
        ah[2][f] = pack_bf16x2(x.x, x.y);
      }
#pragma unroll
      for (int nb2 = 0; nb2 < 2; ++nb2) {
        uint32_t bw[4];
        // matrices: (k 0-7, heads lo), (k 8-15, heads lo), (k 0-7, heads hi), (k 8-15, heads hi)
        ldmatrix_x4_trans(bw, ws + mo_w_off(k0 + (mi & 1) * 8 + (lane & 7), nb2 * 2 + (mi >> 1)));
#pragma unroll
        for (int q = 2; q >= 0; --q) {
          mma_16816(c[2 * nb2], ah[q], bw[0], bw[1]);
          mma_16816(c[2 * nb2 + 1], ah[q], bw[2], bw[3]);
        }
      }
    }
    __syncthreads();                                 // Wo has been read: the sums may take its place
#pragma unroll
    for (int nb = 0; nb < 4; ++nb)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        red[(warp * 16 + g + (e >> 1) * 8) * kMoRedPitch + nb * 8 + 2 * tq + (e & 1)] = c[nb][e];
    __syncthreads();
    if (threadIdx.x < 32 * kTok) {
      // kTok consecutive threads: one head's tokens, which lie side by side in scores and flags
      const int tok = threadIdx.x % kTok, i = i0 + threadIdx.x / kTok, tt = t0 + tok;
      float sc = 0.f;
#pragma unroll
      for (int w = 0; w < kMoWarps; ++w) sc += red[(w * 16 + tok) * kMoRedPitch + threadIdx.x / kTok];
      if (i < h && tt < a.n) {
        const size_t o = ((size_t)b * h + i) * a.n + tt;
        const bool padding = a.seq_lens && tt >= a.seq_lens[b];
        if (scores) scores[o] = sc;
        flags[o] = !padding && (sc + (i0 == 0 ? gamma0 : gamma ? gamma[i] : 0.f)) > logit_tau ? 1 : 0;
      }
    }
  }
}

// Steps of (query tile, key tile) of the whole batch: the list's 32-bit places hold twice this many.
static bool gate_attn_list_fits(const ag_layer_desc &d) {
  const long long nq = (d.seq + kGaBM - 1) / kGaBM;
  return (d.gate_causal ? nq * (nq + 1) : 2 * nq * nq) * d.batch * d.gate_heads < (1LL << 28);
}

bool gate_attn_tc_supported(const ag_layer_desc &d) {
  const int GD = d.gate_heads * d.gate_head_dim;
  if (d.dtype != AG_BF16 || !gate_proj_tc_supported(d.hidden, GD)) return false;
  // Gate heads of 64 have the CUDA-core form for what goes beyond this one: 28 heads, where the output layer alone
  // fits an SM's shared memory and the merge's does not, and prompts of about a million tokens.  (128-wide heads end there.)
  return d.gate_head_dim == 128 ||
         (mo_smem_bytes(GD) + kMoPieceBytes <= kMaxSmemBytes && gate_attn_list_fits(d));
}

// Segments of the list: one per SM.
static int gate_attn_segments(const ag_layer_desc &d, int *n_seg) {
  static int sm_count[64] = {0};                     // per device, read once
  int dev = 0;
  AG_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return AG_ERR_UNSUPPORTED;
  if (sm_count[dev] == 0) {
    int v = 0;
    AG_CUDA_TRY(cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev));
    sm_count[dev] = v < 1 ? 1 : (v > kGaMaxSeg ? kGaMaxSeg : v);
  }
  *n_seg = sm_count[dev];
  return gate_attn_list_fits(d) ? AG_OK : AG_ERR_UNSUPPORTED;
}

size_t gate_attn_partial_bytes(const ag_layer_desc &d) {
  // one slot per piece: query tiles + segments, whatever the device (no device is asked here)
  const size_t nq = (d.seq + kGaBM - 1) / kGaBM;
  const size_t slots = (size_t)d.batch * d.gate_heads * nq + kGaMaxSeg;
  return align_up(slots * kGaBM * d.gate_head_dim * sizeof(float), 256) + align_up(slots * kGaBM * 2 * sizeof(float), 256);
}

template <int kGaD>
static int run_gate_attn_tc(const ag_layer_desc &d, const void *qkv, void *partials,
                            const void *Wo, const float *gamma, float logit_tau, float *scores, uint8_t *flags,
                            cudaStream_t st) {
  constexpr int kGaSmemBytes = GaCfg<kGaD>::kSmemBytes;
  const int GD = d.gate_heads * d.gate_head_dim;
  GateAttnMaps tm;
  int rc;
  const size_t plane = (size_t)d.batch * d.seq * 3 * GD;
  for (int i = 0; i < 3; ++i) {
    const void *part = static_cast<const __nv_bfloat16 *>(qkv) + (i < GaCfg<kGaD>::kParts ? i : 0) * plane;
    if ((rc = make_tmap_3d_bf16(&tm.q[i], part, d.batch, d.seq, 3 * GD, kGaBM, 64))) return rc;
    if ((rc = make_tmap_3d_bf16(&tm.kv[i], part, d.batch, d.seq, 3 * GD, kGaBN, 64))) return rc;
  }
  GateAttnArgs a;
  a.seq_lens = d.seq_lens;
  a.n = d.seq; a.n_qtiles = (d.seq + kGaBM - 1) / kGaBM;
  a.batch = d.batch; a.gate_heads = d.gate_heads; a.GD = GD; a.causal = d.gate_causal;
  if ((rc = gate_attn_segments(d, &a.n_seg))) return rc;
  const size_t slots = (size_t)d.batch * d.gate_heads * a.n_qtiles + kGaMaxSeg;
  a.part_o = static_cast<float *>(partials);
  a.part_ml = reinterpret_cast<float *>(static_cast<char *>(partials) +
                                        align_up(slots * kGaBM * kGaD * sizeof(float), 256));
  a.scale_log2 = (float)(1.4426950408889634 / sqrt((double)kGaD));
  AG_CUDA_TRY(cudaFuncSetAttribute(gate_attn_tc_kernel<kGaD>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGaSmemBytes));
  rc = launch_pdl(gate_attn_tc_kernel<kGaD>, dim3(a.n_seg), dim3(kGaThreads), kGaSmemBytes, st, tm, a);
  if (rc) return rc;
  // fewer tokens per CTA while the CTAs are no more than the SMs (148): an SM then takes in fewer rows of the partials
  const long long tokens = (long long)d.batch * d.seq;
  const int tok = tokens <= 4 * 148 ? 4 : tokens <= 8 * 148 ? 8 : 16;
  auto mo = tok == 4 ? gate_merge_out_kernel<kGaD, 4> : tok == 8 ? gate_merge_out_kernel<kGaD, 8> : gate_merge_out_kernel<kGaD, 16>;
  AG_CUDA_TRY(cudaFuncSetAttribute(mo, cudaFuncAttributeMaxDynamicSharedMemorySize, mo_smem_bytes(GD)));
  const int blocks = d.batch * ((d.seq + tok - 1) / tok);
  return launch_pdl(mo, dim3(blocks), dim3(kMoThreads), mo_smem_bytes(GD), st, a, static_cast<const __nv_bfloat16 *>(Wo),
                    gamma, logit_tau, kv_heads_of(d), scores, flags);
}

int gate_attn_parts(const ag_layer_desc &d) { return d.gate_head_dim == 64 ? GaCfg<64>::kParts : GaCfg<128>::kParts; }

int launch_gate_attn_tc(const ag_layer_desc &d, const void *qkv, void *partials,
                        const void *Wo, const float *gamma, float logit_tau, float *scores, uint8_t *flags,
                        cudaStream_t st) {
  return d.gate_head_dim == 64 ? run_gate_attn_tc<64>(d, qkv, partials, Wo, gamma, logit_tau, scores, flags, st)
                               : run_gate_attn_tc<128>(d, qkv, partials, Wo, gamma, logit_tau, scores, flags, st);
}

int gate_attn_tc_wait_timeouts() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, umma::g_wait_expired, sizeof(int)) != cudaSuccess) return -1;
  return v;
}

}  // namespace ag
