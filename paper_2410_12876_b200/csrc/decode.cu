// Single-query decode attention over the ragged retained cache (Sec. 3.1
// decoding stage; cache = retained tokens only, Sec. 3.3; the new token always
// sees its own key, Eq. 5 case j = t).
//
// Split-K: slab s = (sequence, head) is cut into chunks of rows; a chunk is
// reduced to an un-normalised (o, m, l) triple, and the chunks of a slab are
// merged with the self term (q . k_new, v_new) and normalised.  The work is
// HBM-bound: every cache row is read exactly once with 16-byte vector loads,
// one row per group of kLanes consecutive lanes, several rows in flight per lane.
//
// Two forms.  One thread-block cluster (or one CTA) per slab, the triples merged through distributed shared
// memory - one kernel, no scratch: bf16 nearly always (decode_ctas), float32 up to kClusterMaxSlabs slabs.
// Otherwise decode_partial_kernel writes the triples of up to kMaxSplits chunks per slab to the workspace and
// decode_combine_kernel merges them.
#include <cooperative_groups.h>
#include <math.h>
#include <nvtx3/nvToolsExt.h>

#include <type_traits>

#include "ag_common.cuh"
#include "decode_mma_core.cuh"
#include "launch_rules.cuh"

namespace ag {

constexpr int kMaxSplits = 32;     // chunks per slab the workspace is sized for
constexpr int kPartThreads = 256;
constexpr int kUnroll = 8;         // rows in flight per lane group (x2: K and V)
constexpr int kClusterThreads = 512;    // float32 cluster form: 128 rows in flight per CTA (D = 128)

// Grouped-query attention: slab s = (sequence, query head) of q and o reads the cache slab, k_new
// and v_new of its key/value head.
struct HeadMap {
  int heads, kv_heads;
  __device__ __forceinline__ int kv_slab(int slab) const {
    return (slab / heads) * kv_heads + (slab % heads) / (heads / kv_heads);
  }
};

// The conditional append of the decoding stage (Sec. 3.1 with the gate's flag for the new token),
// for kernels that carry it with the attention of the same step: flag_new = NULL means no append.
struct AppendArgs {
  const uint8_t *flag_new;   // [slabs] or NULL
  const int32_t *cap;
  int32_t *len;
  void *k_rows, *v_rows;
  int32_t *dev_status;
};
// What an append needs to know, asked for ahead of the work of the step: after the barrier that ends it nothing is left
// but the stores (the flag, the capacity, then the row were three trips to L2 in a row at the end of every step).
struct NewRow { uint4 k, v; int64_t row0; int cap; uint32_t on; };    // (as they were read: nothing waits for them here)
// The threads [first, first + row vectors) of ONE CTA per slab carry a row; the others get on = false.
template <typename T, int D>
__device__ __forceinline__ NewRow load_new_row(const AppendArgs &ap, int slab, int64_t row0, const T *k_new,
                                               const T *v_new, int first = 0) {
  constexpr int kVecs = D * (int)sizeof(T) / 16;
  const int vec = (int)threadIdx.x - first;
  NewRow r;
  r.on = 0;
  if (ap.flag_new == nullptr || vec < 0 || vec >= kVecs) return r;
  r.k = ld128(k_new + (size_t)slab * D + vec * (16 / (int)sizeof(T)));
  r.v = ld128(v_new + (size_t)slab * D + vec * (16 / (int)sizeof(T)));
  r.cap = ap.cap[slab];
  r.on = ap.flag_new[slab];
  r.row0 = row0;
  return r;
}
// After every read of len[slab] and of the slab's rows by this launch has completed.  L = the length those reads saw.
template <typename T, int D>
__device__ __forceinline__ void append_new_row(const AppendArgs &ap, const NewRow &r, int slab, int L, int first = 0) {
  if (r.on == 0) return;
  const bool lead = (int)threadIdx.x == first;
  if (L >= r.cap) {
    if (lead && ap.dev_status) atomicOr(ap.dev_status, AG_DEV_OVERFLOW);
    return;
  }
  const size_t dst = (size_t)(r.row0 + L) * D * sizeof(T) + ((int)threadIdx.x - first) * 16;
  *reinterpret_cast<uint4 *>(static_cast<uint8_t *>(ap.k_rows) + dst) = r.k;
  *reinterpret_cast<uint4 *>(static_cast<uint8_t *>(ap.v_rows) + dst) = r.v;
  if (lead) ap.len[slab] = L + 1;
}

// Recent-token window: scores of the query against the ring of its key/value slab, by warps 0 .. n_warps - 1
// of those that call: sm_s[r] = scale_log2 * q . k_r for a live slot (an evicted token the query still
// sees), -inf otherwise.  The caller synchronises the CTA before reading sm_s.
template <typename T, int D>
__device__ __forceinline__ void ring_scores_part(const RecentRing &rg, int kv, const T *q_row,
                                                 float scale_log2, float *sm_s, int warp, int n_warps) {
  const int lane = threadIdx.x & 31;
  for (int r = warp; r < rg.R; r += n_warps) {
    const T *kr = static_cast<const T *>(rg.k) + ((size_t)kv * rg.R + r) * D;
    float a = 0.f;
#pragma unroll
    for (int d = lane; d < D; d += 32) a = fmaf(Elem<T>::load(q_row + d), Elem<T>::load(kr + d), a);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    if (lane == 0) sm_s[r] = rg.live[(size_t)kv * rg.R + r] != 0 ? a * scale_log2 : -INFINITY;
  }
}

template <typename T, int D>
__device__ __forceinline__ void ring_scores(const RecentRing &rg, int kv, const T *q_row,
                                            float scale_log2, float *sm_s) {
  ring_scores_part<T, D>(rg, kv, q_row, scale_log2, sm_s, threadIdx.x >> 5, blockDim.x >> 5);
}

// Rows [r_begin, r_end) of one slab, streamed by a whole CTA of kThreads threads: thread (g, v) =
// (row group, 16-byte slice of the row) ends with its group's running maximum m, sum l and slice
// of o (log2 domain).
template <typename T, int D, int kThreads>
__device__ __forceinline__ void decode_stream_rows(const T *q, const T *k_rows,
                                                   const T *v_rows, int64_t row0, int slab,
                                                   int r_begin, int r_end, float scale_log2, float &m,
                                                   float &l, float (&o)[Elem<T>::kPerVec]) {
  constexpr int kEpl = Elem<T>::kPerVec;        // elements per lane
  constexpr int kLanes = D / kEpl;              // lanes per row
  constexpr int kGroups = kThreads / kLanes;
  const int g = threadIdx.x / kLanes, v = threadIdx.x % kLanes;

  float qf[kEpl];
  Elem<T>::unpack(ld128(q + (size_t)slab * D + v * kEpl), qf);
#pragma unroll
  for (int e = 0; e < kEpl; ++e) qf[e] *= scale_log2;

  const T *Kb = k_rows + (size_t)row0 * D + v * kEpl;
  const T *Vb = v_rows + (size_t)row0 * D + v * kEpl;

  m = -INFINITY; l = 0.f;
#pragma unroll
  for (int e = 0; e < kEpl; ++e) o[e] = 0.f;

  // rows r0 + u * kGroups + g, u < count; rows past r_end are clamped for the load and get weight 0
  auto rows = [&](auto n, int r0) {
    constexpr int count = decltype(n)::value;
    const int r = r0 + g;
    uint4 kv[count], vv[count];
#pragma unroll
    for (int u = 0; u < count; ++u) {
      const int ru = min(r + u * kGroups, r_end - 1);
      kv[u] = ldg128_stream(Kb + (size_t)ru * D);
      vv[u] = ldg128_stream(Vb + (size_t)ru * D);
    }
    float s[count];
#pragma unroll
    for (int u = 0; u < count; ++u) {
      float kf[kEpl];
      Elem<T>::unpack(kv[u], kf);
      float a = 0.f;
#pragma unroll
      for (int e = 0; e < kEpl; ++e) a = fmaf(qf[e], kf[e], a);
#pragma unroll
      for (int off = kLanes / 2; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
      s[u] = (r + u * kGroups < r_end) ? a : -INFINITY;
    }
    float m_new = m;
#pragma unroll
    for (int u = 0; u < count; ++u) m_new = fmaxf(m_new, s[u]);
    // a group may not have seen a valid row yet: keep everything at zero then
    const float alpha = (m_new == -INFINITY) ? 1.f : exp2f(m - m_new);
    l *= alpha;
#pragma unroll
    for (int e = 0; e < kEpl; ++e) o[e] *= alpha;
#pragma unroll
    for (int u = 0; u < count; ++u) {
      const float p = (s[u] == -INFINITY) ? 0.f : exp2f(s[u] - m_new);
      l += p;
      float vf[kEpl];
      Elem<T>::unpack(vv[u], vf);
#pragma unroll
      for (int e = 0; e < kEpl; ++e) o[e] = fmaf(p, vf[e], o[e]);
    }
    m = m_new;
  };
  // The trip counts are the same for every thread of the CTA (the shuffles need whole warps).  A last round of few rows
  // goes in a half or a quarter of a round's registers: the clamped rows' arithmetic was most of a short step.
  // us per step, all rounds whole | so: 4 slabs of 64, 64 rows 3.49 | 2.57, 128 rows 3.50 | 2.87, 256 3.52 | 3.45, 500 4.70 | 4.55, 2000 4.55 | 4.35;
  // 8 slabs of 128, 64 rows 3.28 | 2.66, 256 rows in clusters of eight 4.52 | 3.18, 2000 5.55 | 5.45, 16 of them 4000 11.9 | 11.9.
  // (Skipped row by row instead, full rounds lost: 256 rows of a 512-thread CTA 3.5 -> 3.9 us, 2 x 8 slabs of 500 5.3 -> 7.0.
  // The choice inside the loop of the full rounds cost those 1 - 5 %, and a chunk of the split form - whole rounds, but for a
  // slab's last chunk - pays for any code behind its loop: 512 slabs of 128 with 4000 rows 315 -> 321.)
  constexpr int kRound = kUnroll * kGroups;
  int r0 = r_begin;
  if (kThreads == kPartThreads && (r_end - r_begin) % kRound == 0) {
    for (; r0 < r_end; r0 += kRound) rows(std::integral_constant<int, kUnroll>{}, r0);
    return;
  }
  for (; r_end - r0 > kRound / 2; r0 += kRound) rows(std::integral_constant<int, kUnroll>{}, r0);
  if (r_end - r0 > kRound / 4) rows(std::integral_constant<int, kUnroll / 2>{}, r0);
  else if (r0 < r_end) rows(std::integral_constant<int, kUnroll / 4>{}, r0);
}

template <typename T, int D>
__global__ void __launch_bounds__(kPartThreads)
decode_partial_kernel(const T *q, const T *k_rows,
                      const T *v_rows, const int64_t *row_off,
                      const int32_t *len, float scale_log2, int chunk_rows,
                      float *part_o, float *part_ml, const HeadMap hm) {
  constexpr int kEpl = Elem<T>::kPerVec;
  constexpr int kLanes = D / kEpl;
  constexpr int kGroups = kPartThreads / kLanes;
  const int slab = blockIdx.y, chunk = blockIdx.x;
  const int kv = hm.kv_slab(slab);
  pdl_launch_dependents();
  pdl_wait();
  const int L = len[kv];
  const int r_begin = chunk * chunk_rows;
  if (r_begin >= L) return;
  const int r_end = min(L, r_begin + chunk_rows);
  const int g = threadIdx.x / kLanes, v = threadIdx.x % kLanes;
  float m, l, o[kEpl];
  decode_stream_rows<T, D, kPartThreads>(q, k_rows, v_rows, row_off[kv], slab, r_begin, r_end, scale_log2, m, l, o);

  __shared__ float sm_m[kGroups], sm_l[kGroups];
  __shared__ float sm_o[kGroups][D];
  if (v == 0) { sm_m[g] = m; sm_l[g] = l; }
#pragma unroll
  for (int e = 0; e < kEpl; ++e) sm_o[g][v * kEpl + e] = o[e];
  __syncthreads();
  float mc = -INFINITY;
#pragma unroll
  for (int i = 0; i < kGroups; ++i) mc = fmaxf(mc, sm_m[i]);
  float *po = part_o + ((size_t)slab * kMaxSplits + chunk) * D;
  for (int d = threadIdx.x; d < D; d += kPartThreads) {
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < kGroups; ++i) acc = fmaf(sm_m[i] == -INFINITY ? 0.f : exp2f(sm_m[i] - mc), sm_o[i][d], acc);
    po[d] = acc;
  }
  if (threadIdx.x == 0) {
    float lc = 0.f;
#pragma unroll
    for (int i = 0; i < kGroups; ++i) lc = fmaf(sm_m[i] == -INFINITY ? 0.f : exp2f(sm_m[i] - mc), sm_l[i], lc);
    part_ml[((size_t)slab * kMaxSplits + chunk) * 2 + 0] = mc;
    part_ml[((size_t)slab * kMaxSplits + chunk) * 2 + 1] = lc;
  }
}

// Grouped-query form of the chunk pass: one CTA streams a chunk of a KEY/VALUE slab once for the
// G query heads that share it (G = 2 or 4; rows in flight per lane group halved to make room for
// G running softmaxes per thread) and leaves one triple per query head, where
// decode_combine_kernel expects it.
constexpr int kUnrollGqa = 4;
template <typename T, int D, int G>
__global__ void __launch_bounds__(kPartThreads)
decode_partial_gqa_kernel(const T *q, const T *k_rows,
                          const T *v_rows, const int64_t *row_off,
                          const int32_t *len, float scale_log2, int chunk_rows,
                          float *part_o, float *part_ml, int kv_heads) {
  constexpr int kEpl = Elem<T>::kPerVec;
  constexpr int kLanes = D / kEpl;
  constexpr int kGroups = kPartThreads / kLanes;
  const int kv = blockIdx.y, chunk = blockIdx.x;
  const int slab0 = (kv / kv_heads) * kv_heads * G + (kv % kv_heads) * G;   // first query slab of the group
  pdl_launch_dependents();
  pdl_wait();
  const int L = len[kv];
  const int r_begin = chunk * chunk_rows;
  if (r_begin >= L) return;
  const int r_end = min(L, r_begin + chunk_rows);
  const int g = threadIdx.x / kLanes, v = threadIdx.x % kLanes;

  float qf[G][kEpl], o[G][kEpl], m[G], l[G];
#pragma unroll
  for (int h = 0; h < G; ++h) {
    Elem<T>::unpack(ld128(q + (size_t)(slab0 + h) * D + v * kEpl), qf[h]);
    m[h] = -INFINITY; l[h] = 0.f;
#pragma unroll
    for (int e = 0; e < kEpl; ++e) { qf[h][e] *= scale_log2; o[h][e] = 0.f; }
  }
  const T *Kb = k_rows + (size_t)row_off[kv] * D + v * kEpl;
  const T *Vb = v_rows + (size_t)row_off[kv] * D + v * kEpl;

  // uniform trip count (the shuffles need whole warps); rows past r_end are clamped and get weight 0
  for (int r0 = r_begin; r0 < r_end; r0 += kUnrollGqa * kGroups) {
    const int r = r0 + g;
    uint4 kv4[kUnrollGqa], vv4[kUnrollGqa];
#pragma unroll
    for (int u = 0; u < kUnrollGqa; ++u) {
      const int ru = min(r + u * kGroups, r_end - 1);
      kv4[u] = ldg128_stream(Kb + (size_t)ru * D);
      vv4[u] = ldg128_stream(Vb + (size_t)ru * D);
    }
    float sc[kUnrollGqa][G];
#pragma unroll
    for (int u = 0; u < kUnrollGqa; ++u) {
      float kf[kEpl];
      Elem<T>::unpack(kv4[u], kf);
#pragma unroll
      for (int h = 0; h < G; ++h) {
        float a = 0.f;
#pragma unroll
        for (int e = 0; e < kEpl; ++e) a = fmaf(qf[h][e], kf[e], a);
#pragma unroll
        for (int off = kLanes / 2; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
        sc[u][h] = (r + u * kGroups < r_end) ? a : -INFINITY;
      }
    }
#pragma unroll
    for (int h = 0; h < G; ++h) {
      float m_new = m[h];
#pragma unroll
      for (int u = 0; u < kUnrollGqa; ++u) m_new = fmaxf(m_new, sc[u][h]);
      const float alpha = (m_new == -INFINITY) ? 1.f : exp2f(m[h] - m_new);
      l[h] *= alpha;
#pragma unroll
      for (int e = 0; e < kEpl; ++e) o[h][e] *= alpha;
#pragma unroll
      for (int u = 0; u < kUnrollGqa; ++u) {
        const float p = (sc[u][h] == -INFINITY) ? 0.f : exp2f(sc[u][h] - m_new);
        l[h] += p;
        float vf[kEpl];
        Elem<T>::unpack(vv4[u], vf);
#pragma unroll
        for (int e = 0; e < kEpl; ++e) o[h][e] = fmaf(p, vf[e], o[h][e]);
      }
      m[h] = m_new;
    }
  }

  __shared__ float sm_m[G][kGroups], sm_l[G][kGroups];
  __shared__ float sm_o[kGroups][D];
#pragma unroll
  for (int h = 0; h < G; ++h) {
    __syncthreads();                                 // sm_o of the previous head has been read
    if (v == 0) { sm_m[h][g] = m[h]; sm_l[h][g] = l[h]; }
#pragma unroll
    for (int e = 0; e < kEpl; ++e) sm_o[g][v * kEpl + e] = o[h][e];
    __syncthreads();
    float mc = -INFINITY;
#pragma unroll
    for (int i = 0; i < kGroups; ++i) mc = fmaxf(mc, sm_m[h][i]);
    const size_t slot = (size_t)(slab0 + h) * kMaxSplits + chunk;
    for (int d = threadIdx.x; d < D; d += kPartThreads) {
      float acc = 0.f;
#pragma unroll
      for (int i = 0; i < kGroups; ++i)
        acc = fmaf(sm_m[h][i] == -INFINITY ? 0.f : exp2f(sm_m[h][i] - mc), sm_o[i][d], acc);
      part_o[slot * D + d] = acc;
    }
    if (threadIdx.x == 0) {
      float lc = 0.f;
#pragma unroll
      for (int i = 0; i < kGroups; ++i) lc = fmaf(sm_m[h][i] == -INFINITY ? 0.f : exp2f(sm_m[h][i] - mc), sm_l[h][i], lc);
      part_ml[slot * 2 + 0] = mc;
      part_ml[slot * 2 + 1] = lc;
    }
  }
}

// Merges the chunks' triples of every query slab with the self term.  CTA (slab, y): D threads
// (thread d owns output dimension d) for each of blockDim.y query heads of the key/value slab's group.  One CTA per slab
// where it appends, which then is the only one that reads the slab's length; else as many as the group fills (in one CTA, eight
// rounds for 32 heads, a step of 4 such slabs took 35 us, 21 with an append of its own).  The chunks' weights are computed
// side by side, a chunk per lane, and the partial outputs are loaded eight at a time: one chunk after the
// other, each load waiting for its turn, took 11.5 us for 1024 query slabs of 17 chunks.
__host__ __device__ constexpr int combine_heads(int D) { return 512 / D; }     // query heads at once
template <typename T, int D>
__global__ void __launch_bounds__(512)
decode_combine_kernel(const T *q, const T *k_new,
                      const T *v_new, const int32_t *len,
                      float scale_log2, int chunk_rows, const float *part_o,
                      const float *part_ml, T *o,
                      const int64_t *row_off, int G, const AppendArgs ap, const RecentRing rg) {
  static_assert(kMaxSplits == 32, "a lane per chunk");
  const int kv = blockIdx.x, d = threadIdx.x, y = threadIdx.y, lane = d & 31;
  constexpr int kMaxHeads = combine_heads(D);
  __shared__ float red[kMaxHeads][D / 32];
  __shared__ float ring_s[kMaxHeads][kMaxRecent];
  __shared__ float wgt[kMaxHeads][kMaxSplits];       // weight of every chunk
  __shared__ float lsum_s[kMaxHeads][2];             // maximum and sum over chunks, self and ring
  pdl_launch_dependents();
  pdl_wait();
  const float kn = Elem<T>::load(k_new + (size_t)kv * D + d), vn = Elem<T>::load(v_new + (size_t)kv * D + d);
  const int L = len[kv];
  NewRow row;
  row.on = 0;
  if (y == 0) row = load_new_row<T, D>(ap, kv, row_off[kv], k_new, v_new);
  const int n_chunks = (L + chunk_rows - 1) / chunk_rows;
  for (int h0 = blockIdx.y * blockDim.y; h0 < G; h0 += gridDim.y * blockDim.y) {
    const int h = h0 + y;
    const bool on = h < G;                           // whole warps: D is a multiple of 32
    const int slab = kv * G + min(h, G - 1);
    float a = Elem<T>::load(q + (size_t)slab * D + d) * kn;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
    if (lane == 0) red[y][d >> 5] = a;
    ring_scores_part<T, D>(rg, kv, q + (size_t)slab * D, scale_log2, ring_s[y], d >> 5, D / 32);
    __syncthreads();
    if (d < 32) {
      // one warp per head: the chunks' maxima and sums, one per lane
      float s_self = 0.f;
#pragma unroll
      for (int i = 0; i < D / 32; ++i) s_self += red[y][i];
      s_self *= scale_log2;
      const float2 ml = lane < n_chunks ? *reinterpret_cast<const float2 *>(part_ml + ((size_t)slab * kMaxSplits + lane) * 2)
                                        : make_float2(-INFINITY, 0.f);
      const float rs = lane < rg.R ? ring_s[y][lane] : -INFINITY;
      float m = fmaxf(fmaxf(ml.x, rs), s_self);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
      const float w = exp2f(ml.x - m), wr = exp2f(rs - m);      // 2^-inf = 0
      float l = fmaf(w, ml.y, wr);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) l += __shfl_xor_sync(0xffffffffu, l, off);
      wgt[y][lane] = w;
      if (lane < rg.R) ring_s[y][lane] = wr;
      if (lane == 0) {
        const float w_self = exp2f(s_self - m);
        lsum_s[y][0] = w_self;
        lsum_s[y][1] = l + w_self;
      }
    }
    __syncthreads();
    float acc = lsum_s[y][0] * vn;
    const float *po = part_o + (size_t)slab * kMaxSplits * D + d;
    for (int c0 = 0; c0 < n_chunks; c0 += 8) {
      float x[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) x[c] = c0 + c < n_chunks ? po[(size_t)(c0 + c) * D] : 0.f;
#pragma unroll
      for (int c = 0; c < 8; ++c) acc = fmaf(wgt[y][c0 + c], x[c], acc);
    }
    // the evicted tokens of the recent-token window
    for (int r = 0; r < rg.R; ++r) {
      const float w = ring_s[y][r];
      if (w > 0.f) acc = fmaf(w, Elem<T>::load(static_cast<const T *>(rg.v) + ((size_t)kv * rg.R + r) * D + d), acc);
    }
    if (on) Elem<T>::store(o + (size_t)slab * D + d, acc / lsum_s[y][1]);
    __syncthreads();                                 // shared memory of this round has been read
  }
  // Every thread of the CTA has read the slab's length, and the chunk pass, the only reader of the slab's
  // rows, has completed: the new row may go in and the length may move; the ring has been read too.
  if (y == 0) {
    append_new_row<T, D>(ap, row, kv, L);
    constexpr int kVecs = D * (int)sizeof(T) / 16;
    if (rg.R > 0 && ap.flag_new != nullptr && d < kVecs)
      ring_put<kVecs>(rg, kv, d, reinterpret_cast<const uint8_t *>(k_new + (size_t)kv * D),
                      reinterpret_cast<const uint8_t *>(v_new + (size_t)kv * D), ap.flag_new[kv] != 0);
  }
}

// One cluster of kClusterSize CTAs per slab.  CTA `rank` reduces rows [rank, rank + 1) * per of
// the slab to a triple in its own shared memory; after a cluster barrier the first CTA reads all
// triples through distributed shared memory, adds the self term and writes the output.  The
// second barrier keeps every CTA's shared memory alive until it has been read.  No CTA leaves
// early: the cluster barriers need all of them.
//
// kCtas = 1: a cluster of one, for caches that one CTA streams in a round or two (its barriers are the CTA's own).
template <typename T, int D, int kThreads, int kCtas>
__global__ void __launch_bounds__(kThreads, 2)
decode_cluster_kernel(const T *q, const T *k_new, const T *v_new,
                      const T *k_rows, const T *v_rows,
                      const int64_t *row_off, const int32_t *len,
                      float scale_log2, T *out, const AppendArgs ap, const HeadMap hm,
                      const RecentRing rg) {
  namespace cg = cooperative_groups;
  constexpr int kEpl = Elem<T>::kPerVec;
  constexpr int kLanes = D / kEpl;
  constexpr int kGroups = kThreads / kLanes;
  cg::cluster_group cluster = cg::this_cluster();
  const int slab = blockIdx.y, rank = kCtas == 1 ? 0 : (int)cluster.block_rank();
  const int kv = hm.kv_slab(slab);
  pdl_launch_dependents();
  pdl_wait();
  const int L = len[kv];
  const int per = ((L + kCtas - 1) / kCtas + kGroups - 1) / kGroups * kGroups;
  const int r_begin = min(L, rank * per), r_end = min(L, r_begin + per);
  const int g = threadIdx.x / kLanes, v = threadIdx.x % kLanes;

  __shared__ float sm_m[kGroups], sm_l[kGroups];
  __shared__ float sm_o[kGroups][D];
  __shared__ float cta_o[D];          // this CTA's triple, read by the first CTA of the cluster
  __shared__ float cta_ml[2];
  __shared__ float red[D / 32];
  __shared__ float ring_s[kMaxRecent];

  // self score q . k_new: only the first CTA needs it; its loads are in flight with the stream's
  // (and the new value, which the merge after the cluster barrier would otherwise wait for)
  T q_raw = T(0.f), k_raw = T(0.f), v_raw = T(0.f);    // (not used before the stream is done)
  if (rank == 0 && threadIdx.x < D) {
    q_raw = q[(size_t)slab * D + threadIdx.x];
    k_raw = k_new[(size_t)kv * D + threadIdx.x];
    v_raw = v_new[(size_t)kv * D + threadIdx.x];
  }

  float m, l, o[kEpl];
  decode_stream_rows<T, D, kThreads>(q, k_rows, v_rows, row_off[kv], slab, r_begin, r_end, scale_log2, m, l, o);

  if (v == 0) { sm_m[g] = m; sm_l[g] = l; }
#pragma unroll
  for (int e = 0; e < kEpl; ++e) sm_o[g][v * kEpl + e] = o[e];
  const float v_self = Elem<T>::load(&v_raw);
  if (threadIdx.x < D) {              // whole warps: D is a multiple of 32
    float prod = Elem<T>::load(&q_raw) * Elem<T>::load(&k_raw);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) prod += __shfl_xor_sync(0xffffffffu, prod, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = prod;
  }
  if (rank == 0) ring_scores<T, D>(rg, kv, q + (size_t)slab * D, scale_log2, ring_s);
  __syncthreads();
  float mc = -INFINITY;
#pragma unroll
  for (int i = 0; i < kGroups; ++i) mc = fmaxf(mc, sm_m[i]);
  if (threadIdx.x < D) {
    float acc = 0.f;
#pragma unroll
    for (int i = 0; i < kGroups; ++i)
      acc = fmaf(sm_m[i] == -INFINITY ? 0.f : exp2f(sm_m[i] - mc), sm_o[i][threadIdx.x], acc);
    cta_o[threadIdx.x] = acc;
  }
  if (threadIdx.x == 0) {
    float lc = 0.f;
#pragma unroll
    for (int i = 0; i < kGroups; ++i) lc = fmaf(sm_m[i] == -INFINITY ? 0.f : exp2f(sm_m[i] - mc), sm_l[i], lc);
    cta_ml[0] = mc;
    cta_ml[1] = lc;
  }
  if constexpr (kCtas > 1) cluster.sync();
  else __syncthreads();
  // every CTA of the cluster has read the length and its rows: the new row may go in
  // (never asked for when query heads share a slab: another head's cluster may still be reading its length)
  // by threads that have no part in the merge below, so that the two run side by side (asked for any earlier, the row
  // is waited for at this barrier: 95 -> 105 us for a 128-token float32 layer and 16 steps)
  if (rank == 0) append_new_row<T, D>(ap, load_new_row<T, D>(ap, kv, row_off[kv], k_new, v_new, D), kv, L, D);
  if (rank == 0 && threadIdx.x < D) {
    const int d = threadIdx.x;
    float s_self = 0.f;
#pragma unroll
    for (int i = 0; i < D / 32; ++i) s_self += red[i];
    s_self *= scale_log2;
    float mr[kCtas], lr[kCtas], orr[kCtas];
#pragma unroll
    for (int r = 0; r < kCtas; ++r) {
      const float *ml = kCtas == 1 ? cta_ml : cluster.map_shared_rank(cta_ml, r);
      mr[r] = ml[0];
      lr[r] = ml[1];
      orr[r] = (kCtas == 1 ? cta_o : cluster.map_shared_rank(cta_o, r))[d];
    }
    float mm = s_self;
#pragma unroll
    for (int r = 0; r < kCtas; ++r) mm = fmaxf(mm, mr[r]);
    for (int r = 0; r < rg.R; ++r) mm = fmaxf(mm, ring_s[r]);
    const float w_self = exp2f(s_self - mm);
    float acc = w_self * v_self;
    float lsum = w_self;
#pragma unroll
    for (int r = 0; r < kCtas; ++r) {
      const float w = mr[r] == -INFINITY ? 0.f : exp2f(mr[r] - mm);
      acc = fmaf(w, orr[r], acc);
      lsum = fmaf(w, lr[r], lsum);
    }
    // the evicted tokens of the recent-token window
    for (int r = 0; r < rg.R; ++r) {
      if (ring_s[r] == -INFINITY) continue;
      const float w = exp2f(ring_s[r] - mm);
      acc = fmaf(w, Elem<T>::load(static_cast<const T *>(rg.v) + ((size_t)kv * rg.R + r) * D + d), acc);
      lsum += w;
    }
    Elem<T>::store(out + (size_t)slab * D + d, acc / lsum);
  }
  if (rank == 0 && rg.R > 0 && ap.flag_new != nullptr) {
    // the step carries the append: the new token joins the ring once every thread has read it
    constexpr int kVecs = D * (int)sizeof(T) / 16;
    __syncthreads();
    if ((int)threadIdx.x < kVecs)
      ring_put<kVecs>(rg, kv, threadIdx.x, reinterpret_cast<const uint8_t *>(k_new + (size_t)kv * D),
                      reinterpret_cast<const uint8_t *>(v_new + (size_t)kv * D), ap.flag_new[kv] != 0);
  }
  if constexpr (kCtas > 1) cluster.sync();
}

// The cluster form for bf16, with the rows streamed through shared memory and the scores and weighted sums
// on warp-level MMAs (decode_mma_core.cuh): per row a fraction of the instructions of the CUDA-core form,
// which at these sizes is bound by instruction issue and by what one SM can take in, not by latency alone.
// One cluster per run of G <= 16 query slabs that share a key/value slab (G = 1 without grouped-query
// attention): the G queries are columns of one MMA operand, so the slab is read once for all of them, and the
// one cluster that reads it may append to it.  CTA `rank` takes whole 64-row tiles; after the cluster
// barrier rank r merges the heads r, r + kCtas, ... of the group, whose triples the ranks have written to its shared memory.
// Nothing of the cache is read ahead of the wait for the preceding kernel, which may be one that lays it out: where a
// slab begins arrives with its length, the queries in the same trip (the queries behind the length: 127.5 -> 133.6 us for
// 16 steps; the first tile asked for from where the slab seemed to lie before the wait, checked after it: 131.3).
// A step of 32 slabs of 400 .. 1640 rows takes 7.8 us in a graph (1.2 us of it an empty chain of launches); it was 9.2 us
// with the queries as the rows of the MMAs, the merging rank reading the others' triples (one trip and one barrier
// more), the row to append fetched after the barrier and 96 KB of stages: two stages and fewer than 170 registers let
// three CTAs share an SM, so the next step's clusters start beside this one's.
constexpr int kCmStages = 2;
// kMaxG: 1 (one query per slab), 4, 8 or 16.  kCtas: CTAs of a cluster (1: no cluster).
template <int D, int kMaxG, int kCtas>
__global__ void __launch_bounds__(kGqThreads, 2)
decode_cluster_mma_kernel(const __nv_bfloat16 *q, const __nv_bfloat16 *k_new,
                          const __nv_bfloat16 *v_new, const __nv_bfloat16 *k_rows,
                          const __nv_bfloat16 *v_rows, const int64_t *row_off,
                          const int32_t *len, float scale_log2, __nv_bfloat16 *out, int group,
                          const AppendArgs ap, const HeadMap hm, const RecentRing rg) {
  namespace cg = cooperative_groups;
  using T = __nv_bfloat16;
  static_assert(kGqThreads >= D, "one thread per output dimension in the merge");
  constexpr int kHeads = (kMaxG + kCtas - 1) / kCtas;    // heads a rank merges, at most
  const int G = kMaxG == 1 ? 1 : group;
  extern __shared__ __align__(128) uint8_t gq_smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int slab0 = blockIdx.y * G, rank = kCtas == 1 ? 0 : (int)cluster.block_rank();
  const int kv = hm.kv_slab(slab0);
  const int d = threadIdx.x;
  pdl_launch_dependents();
  if constexpr (kCtas > 1) cluster.barrier_arrive();   // (waited for before the first write to another rank: all have started then)
  pdl_wait();
  const int L = len[kv];
  const int64_t slab_row0 = row_off[kv];
  const int r_first = rank * kGqTile;
  const GqQuery<D, kMaxG> qf = gq_load_query<D, kMaxG>(q + (size_t)slab0 * D, G);

  // the ranks' triples of the heads this rank merges, written by the ranks themselves
  __shared__ float in_o[kHeads][kCtas][D];
  __shared__ float2 in_ml[kHeads][kCtas];
  auto at_rank = [&](auto *p, int r) { return kCtas == 1 ? p : cluster.map_shared_rank(p, r); };
  __shared__ float red[kHeads][D / 32];
  __shared__ float ring_s[kHeads][kMaxRecent];

  // self scores q . k_new of the heads this rank merges, and the new value: in flight with the stream
  T q_raw[kHeads], k_raw = T(0.f), v_raw = T(0.f);           // (not used before the stream is done)
#pragma unroll
  for (int u = 0; u < kHeads; ++u) {
    const int h = rank + u * kCtas;
    q_raw[u] = (h < G && d < D) ? q[(size_t)(slab0 + h) * D + d] : T(0.f);
  }
  if (rank < G && d < D) {
    k_raw = k_new[(size_t)kv * D + d];
    v_raw = v_new[(size_t)kv * D + d];
  }
  NewRow row;
  row.on = 0;
  if (rank == 0) row = load_new_row<T, D>(ap, kv, slab_row0, k_new, v_new);

  const uint8_t *Kg = reinterpret_cast<const uint8_t *>(k_rows) + (size_t)slab_row0 * (D * 2);
  const uint8_t *Vg = reinterpret_cast<const uint8_t *>(v_rows) + (size_t)slab_row0 * (D * 2);
  if (r_first < L) {                  // the same for the whole CTA
    const GqWarpTriples w = gq_stream_rows<D, kCmStages, kMaxG>(gq_smem, qf, G, Kg, Vg, r_first, kCtas * kGqTile, L,
                                                                scale_log2);
    if constexpr (kCtas > 1) cluster.barrier_wait();
    for (int x = d; x < G * D; x += kGqThreads) {
      const int h = x / D, e = x % D, to = h % kCtas;
      float acc, mc, lc;
      gq_combine<D>(w, h, e, acc, mc, lc);
      *at_rank(&in_o[h / kCtas][rank][e], to) = acc;
      if (e == 0) *at_rank(&in_ml[h / kCtas][rank], to) = make_float2(mc, lc);
    }
  } else {
    if constexpr (kCtas > 1) cluster.barrier_wait();
    // weight 0 in the merge, which then skips the values
    if (d < G) *at_rank(&in_ml[d / kCtas][rank], d % kCtas) = make_float2(-INFINITY, 0.f);
  }
#pragma unroll
  for (int u = 0; u < kHeads; ++u) {
    const int h = rank + u * kCtas;
    if (h >= G) break;                // the same for the whole CTA
    float prod = Elem<T>::load(&q_raw[u]) * Elem<T>::load(&k_raw);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) prod += __shfl_xor_sync(0xffffffffu, prod, off);
    if ((d & 31) == 0 && d < D) red[u][d >> 5] = prod;
    ring_scores<T, D>(rg, kv, q + (size_t)(slab0 + h) * D, scale_log2, ring_s[u]);
  }
  const float v_self = Elem<T>::load(&v_raw);
  if constexpr (kCtas > 1) cluster.sync();
  else __syncthreads();
  // every CTA of the cluster has read the length and its rows: the new row may go in
  // (never asked for when a query slab outside this cluster shares the slab)
  if (rank == 0) append_new_row<T, D>(ap, row, kv, L);
#pragma unroll
  for (int u = 0; u < kHeads; ++u) {
    const int h = rank + u * kCtas;
    if (h >= G || d >= D) break;
    float s_self = 0.f;
#pragma unroll
    for (int i = 0; i < D / 32; ++i) s_self += red[u][i];
    s_self *= scale_log2;
    float mm = s_self;
#pragma unroll
    for (int r = 0; r < kCtas; ++r) mm = fmaxf(mm, in_ml[u][r].x);
    for (int r = 0; r < rg.R; ++r) mm = fmaxf(mm, ring_s[u][r]);
    const float w_self = exp2f(s_self - mm);
    float acc = w_self * v_self;
    float lsum = w_self;
#pragma unroll
    for (int r = 0; r < kCtas; ++r) {
      const float2 ml = in_ml[u][r];
      if (ml.x == -INFINITY) continue;                 // a rank without rows has sent no values
      const float w = exp2f(ml.x - mm);
      acc = fmaf(w, in_o[u][r][d], acc);
      lsum = fmaf(w, ml.y, lsum);
    }
    // the evicted tokens of the recent-token window
    for (int r = 0; r < rg.R; ++r) {
      if (ring_s[u][r] == -INFINITY) continue;
      const float w = exp2f(ring_s[u][r] - mm);
      acc = fmaf(w, Elem<T>::load(static_cast<const T *>(rg.v) + ((size_t)kv * rg.R + r) * D + d), acc);
      lsum += w;
    }
    Elem<T>::store(out + (size_t)(slab0 + h) * D + d, acc / lsum);
  }
  if (rg.R > 0 && ap.flag_new != nullptr) {
    // the step carries the append: the new token joins the ring once every rank has read it
    if constexpr (kCtas > 1) cluster.sync();
    else __syncthreads();
    constexpr int kVecs = D * (int)sizeof(T) / 16;
    if (rank == 0 && d < kVecs)
      ring_put<kVecs>(rg, kv, d, reinterpret_cast<const uint8_t *>(k_new + (size_t)kv * D),
                      reinterpret_cast<const uint8_t *>(v_new + (size_t)kv * D), ap.flag_new[kv] != 0);
  }
}

template <int D, int kMaxG, int kCtas>
static cudaLaunchConfig_t cluster_mma_config(int groups, cudaStream_t st, cudaLaunchAttribute *attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCtas, groups);
  cfg.blockDim = dim3(kGqThreads);
  cfg.dynamicSmemBytes = gq_smem_bytes(D, kCmStages);
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCtas; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1] = pdl_attribute();
  cfg.attrs = kCtas == 1 ? attr + 1 : attr;
  cfg.numAttrs = kCtas == 1 ? 1 : 2;
  return cfg;
}

// A kernel that leaves no room for another CTA on its SM, to ask how many clusters have an SM for each of their CTAs.
constexpr int kAloneSmem = 120 * 1024;
__global__ void __launch_bounds__(kGqThreads) decode_alone_kernel() {}

// Clusters of `ctas` CTAs of `kern` that the device holds at once, 0 where it cannot place one (more than eight are not portable:
// part of a device, or a context with few SMs).  Sets the kernel's attributes.
static int clusters_at_once(const void *kern, cudaLaunchConfig_t cfg, cudaLaunchAttribute *attr, int ctas, size_t smem) {
  cfg.gridDim.x = attr[0].val.clusterDim.x = ctas;
  cfg.dynamicSmemBytes = smem;
  int n = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess &&
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess)
    return n;
  (void)cudaGetLastError();
  return 0;
}

// Asked for once per thread and context; the attributes of the kernels of more than eight CTAs are set then.
template <int D, int kMaxG>
static DecodePlaces decode_places() {
  struct Answer { unsigned long long context; DecodePlaces places; };
  static thread_local Answer known[8] = {};
  const unsigned long long context = current_context();
  Answer &a = known[context % 8];
  if (context == 0 || a.context != context) {
    const void *alone = reinterpret_cast<const void *>(&decode_alone_kernel);
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = cluster_mma_config<D, kMaxG, kWideCluster>(1, nullptr, attr);
    const size_t smem = cfg.dynamicSmemBytes;
    a.places.wide = clusters_at_once(reinterpret_cast<const void *>(&decode_cluster_mma_kernel<D, kMaxG, kWideCluster>), cfg, attr, kWideCluster, smem);
    a.places.wide_apart = a.places.wide > 0 ? clusters_at_once(alone, cfg, attr, kWideCluster, kAloneSmem) : 0;
    a.places.ten_apart = 0;
    if constexpr (kMaxG <= 4)
      if (clusters_at_once(reinterpret_cast<const void *>(&decode_cluster_mma_kernel<D, kMaxG, kTenCluster>), cfg, attr, kTenCluster, smem) > 0)
        a.places.ten_apart = clusters_at_once(alone, cfg, attr, kTenCluster, kAloneSmem);
    a.context = context;
  }
  return a.places;
}

// groups: clusters (runs of G query slabs on one key/value slab each)
template <int D, int kMaxG, int kCtas>
static int launch_decode_cluster_mma(int groups, int G, const void *q, const void *k_new, const void *v_new,
                                     const ag_cache &c, float scale_log2, void *o, const AppendArgs &ap,
                                     const HeadMap &hm, const RecentRing &rg, cudaStream_t st) {
  using T = __nv_bfloat16;
  if constexpr (kCtas <= kClusterSize)               // (the larger ones': decode_places)
    AG_CUDA_TRY(cudaFuncSetAttribute(decode_cluster_mma_kernel<D, kMaxG, kCtas>, cudaFuncAttributeMaxDynamicSharedMemorySize, gq_smem_bytes(D, kCmStages)));
  cudaLaunchAttribute attr[2];
  const cudaLaunchConfig_t cfg = cluster_mma_config<D, kMaxG, kCtas>(groups, st, attr);
  AG_CUDA_TRY(cudaLaunchKernelEx(&cfg, decode_cluster_mma_kernel<D, kMaxG, kCtas>, static_cast<const T *>(q),
                                 static_cast<const T *>(k_new), static_cast<const T *>(v_new),
                                 static_cast<const T *>(c.k_rows), static_cast<const T *>(c.v_rows),
                                 c.row_off, c.len, scale_log2, static_cast<T *>(o), G, ap, hm, rg));
  return AG_OK;
}

template <typename T, int D, int kThreads, int kCtas>
static int launch_decode_cluster(int slabs, const void *q, const void *k_new, const void *v_new,
                                 const ag_cache &c, float scale_log2, void *o, const AppendArgs &ap,
                                 const HeadMap &hm, const RecentRing &rg, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kCtas, slabs);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCtas; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1] = pdl_attribute();
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  AG_CUDA_TRY(cudaLaunchKernelEx(&cfg, decode_cluster_kernel<T, D, kThreads, kCtas>, static_cast<const T *>(q),
                                 static_cast<const T *>(k_new), static_cast<const T *>(v_new),
                                 static_cast<const T *>(c.k_rows), static_cast<const T *>(c.v_rows),
                                 c.row_off, c.len, scale_log2, static_cast<T *>(o), ap, hm, rg));
  return AG_OK;
}

size_t decode_workspace_bytes(const ag_layer_desc &d) {
  const size_t slabs = (size_t)d.batch * d.heads;
  return align_up(slabs * kMaxSplits * (d.head_dim + 2) * sizeof(float), 256);
}

// Whether the kernels a decode step takes can carry the append: whichever CTA or cluster appends to a slab has to be the
// only one that reads it.  Not so where query heads that share a slab go to clusters of their own, or are more than a CTA
// of the merge takes at once.
static bool decode_carries_append(const ag_layer_desc &d, const ag_cache &c) {
  const int slabs = d.batch * d.heads, group = d.heads / kv_heads_of(d);
  if (group == 1) return true;
  const bool grouped = d.dtype == AG_BF16 && group <= kGqMaxGroup;        // one cluster per key/value slab
  if (slabs <= kClusterMaxSlabs) return grouped;
  const int ctas = !grouped ? 0 : decode_ctas(d.head_dim, slabs / group, slabs, group, c.max_cap, DecodePlaces{});
  return ctas > 0 || group <= combine_heads(d.head_dim);
}

template <typename T, int D>
static int run_decode(const ag_layer_desc &d, const void *q, const void *k_new, const void *v_new,
                      const ag_cache &c, float scale, void *o, void *ws, const AppendArgs &ap, cudaStream_t st) {
  const int slabs = d.batch * d.heads;              // one per (sequence, query head)
  const HeadMap hm{d.heads, kv_heads_of(d)};
  const int group = hm.heads / hm.kv_heads, kv_slabs = d.batch * hm.kv_heads;
  const RecentRing rg = ring_of(d, c);
  const float scale_log2 = scale * 1.4426950408889634f;
  if constexpr (std::is_same_v<T, __nv_bfloat16>) {
    // grouped-query attention: one cluster per key/value slab reads it for all its query heads
    auto cluster = [&](auto ctas, int groups, int G) {
      constexpr int kCtas = decltype(ctas)::value;
      constexpr int kMost = kCtas == kTenCluster ? 4 : 16;             // heads
      return (G == 1 ? launch_decode_cluster_mma<D, 1, kCtas> : G <= 4 ? launch_decode_cluster_mma<D, 4, kCtas> :
              G <= 8 ? launch_decode_cluster_mma<D, kMost < 8 ? kMost : 8, kCtas> : launch_decode_cluster_mma<D, kMost, kCtas>)(groups, G, q, k_new, v_new, c, scale_log2, o, ap, hm, rg, st);
    };
    const int n = group <= kGqMaxGroup ? kv_slabs : slabs, G = group <= kGqMaxGroup ? group : 1;
    // (clusters of one query head each never carry the append: see decode_carries_append)
    const DecodePlaces places = n > kWideMaxSlabs ? DecodePlaces{} : G == 1 ? decode_places<D, 1>() : G <= 4 ? decode_places<D, 4>() :
                                G <= 8 ? decode_places<D, 8>() : decode_places<D, 16>();
    switch (group <= kGqMaxGroup || n <= kClusterMaxSlabs ? decode_ctas(D, n, slabs, G, c.max_cap, places) : 0) {
      case 1: return cluster(std::integral_constant<int, 1>{}, n, G);
      case 2: return cluster(std::integral_constant<int, 2>{}, n, G);
      case 4: return cluster(std::integral_constant<int, 4>{}, n, G);
      case 8: return cluster(std::integral_constant<int, 8>{}, n, G);
      case kTenCluster: return cluster(std::integral_constant<int, kTenCluster>{}, n, G);
      case kWideCluster: return cluster(std::integral_constant<int, kWideCluster>{}, n, G);
    }
  } else {
    // caches of at most two rounds of one CTA's rows (host-known bound): no cluster
    constexpr int kRound = kUnroll * kClusterThreads / (D / Elem<T>::kPerVec);
    if (slabs <= kClusterMaxSlabs)
      return (c.max_cap <= 2 * kRound ? launch_decode_cluster<T, D, kClusterThreads, 1>
                                      : launch_decode_cluster<T, D, kClusterThreads, kClusterSize>)(slabs, q, k_new, v_new, c, scale_log2, o, ap, hm, rg, st);
  }
  int chunk_rows = (c.max_cap + kMaxSplits - 1) / kMaxSplits;
  chunk_rows = (chunk_rows + 127) / 128 * 128;   // whole iterations of the partial kernel (bf16, D = 128)
  const int n_chunks = c.max_cap > 0 ? (c.max_cap + chunk_rows - 1) / chunk_rows : 0;
  float *part_o = static_cast<float *>(ws);
  float *part_ml = part_o + (size_t)slabs * kMaxSplits * D;
  auto qp = static_cast<const T *>(q), kn = static_cast<const T *>(k_new), vn = static_cast<const T *>(v_new);
  auto kr = static_cast<const T *>(c.k_rows), vr = static_cast<const T *>(c.v_rows);
  int rc = AG_OK;
  if (n_chunks > 0 && decode_gqa_mma_supported(d)) {
    // grouped-query attention, bf16: the group's heads are the columns of the MMAs
    rc = launch_decode_partial_gqa_mma(d, q, c, scale_log2, chunk_rows, n_chunks, part_o, part_ml, kMaxSplits, st);
  } else if (std::is_same_v<T, float> && n_chunks > 0 && (group == 2 || group == 4)) {
    // grouped-query attention: the rows of a key/value slab are read once for its query heads
    if constexpr (std::is_same_v<T, float>)
      rc = launch_pdl(group == 2 ? decode_partial_gqa_kernel<T, D, 2> : decode_partial_gqa_kernel<T, D, 4>,
                      dim3(n_chunks, kv_slabs), dim3(kPartThreads), 0, st, qp, kr, vr, c.row_off, c.len, scale_log2,
                      chunk_rows, part_o, part_ml, hm.kv_heads);
  } else if (n_chunks > 0) {
    rc = launch_pdl(decode_partial_kernel<T, D>, dim3(n_chunks, slabs), dim3(kPartThreads), 0, st, qp, kr, vr, c.row_off,
                    c.len, scale_log2, chunk_rows, part_o, part_ml, hm);
  }
  if (rc) return rc;
  const int heads = group < combine_heads(D) ? group : combine_heads(D);
  return launch_pdl(decode_combine_kernel<T, D>, dim3(kv_slabs, ap.flag_new ? 1 : (group + heads - 1) / heads), dim3(D, heads), 0, st, qp, kn,
                    vn, c.len, scale_log2, chunk_rows, part_o, part_ml, static_cast<T *>(o), c.row_off, group, ap, rg);
}

static int dispatch_decode(const ag_layer_desc &d, const void *q, const void *k_new, const void *v_new,
                           const ag_cache &c, float scale, void *o, void *ws, const AppendArgs &ap,
                           cudaStream_t st) {
  if (d.dtype == AG_F32) {
    if (d.head_dim == 64) return run_decode<float, 64>(d, q, k_new, v_new, c, scale, o, ws, ap, st);
    return run_decode<float, 128>(d, q, k_new, v_new, c, scale, o, ws, ap, st);
  }
  if (d.head_dim == 64) return run_decode<__nv_bfloat16, 64>(d, q, k_new, v_new, c, scale, o, ws, ap, st);
  return run_decode<__nv_bfloat16, 128>(d, q, k_new, v_new, c, scale, o, ws, ap, st);
}

int launch_decode(const ag_layer_desc &d, const void *q, const void *k_new, const void *v_new,
                  const ag_cache &c, float scale, void *o, void *ws, size_t, cudaStream_t st) {
  return dispatch_decode(d, q, k_new, v_new, c, scale, o, ws, AppendArgs{}, st);
}

// Attention of the step and the conditional append in the same launches.
int launch_decode_step(const ag_layer_desc &d, const void *q, const void *k_new, const void *v_new,
                       const uint8_t *flag_new, const ag_cache &c, float scale, void *o,
                       int32_t *dev_status, void *ws, cudaStream_t st) {
  if (!decode_carries_append(d, c)) {
    // query heads share a slab: the append waits for all of them, in a launch of its own
    int rc = dispatch_decode(d, q, k_new, v_new, c, scale, o, ws, AppendArgs{}, st);
    if (rc) return rc;
    return launch_append(d, k_new, v_new, flag_new, c, dev_status, st);
  }
  AppendArgs ap;
  ap.flag_new = flag_new; ap.cap = c.cap; ap.len = c.len;
  ap.k_rows = c.k_rows; ap.v_rows = c.v_rows; ap.dev_status = dev_status;
  return dispatch_decode(d, q, k_new, v_new, c, scale, o, ws, ap, st);
}

// ---------------------------------------------------------------------------
// ag_decode_attn_noalloc: decode attention whose split-K scratch is a fixed
// array inside the library, for callers that cannot obtain device memory.
// ---------------------------------------------------------------------------
constexpr size_t kNoAllocScratchBytes = (size_t)1024 * kMaxSplits * (128 + 2) * sizeof(float);  // 17,039,360

// Lives in the global memory of every GPU that loads the library, until exit.
// Host code may only use this name to look the device address up.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

// Device address of g_noalloc_scratch on the CURRENT device, looked up once per device.
static int noalloc_scratch_ptr(void **out) {
  constexpr int kMaxDevices = 64;
  static void *ptrs[kMaxDevices] = {};
  int dev = -1;
  AG_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return AG_ERR_UNSUPPORTED;
  void *p = __atomic_load_n(&ptrs[dev], __ATOMIC_ACQUIRE);
  if (!p) {
    AG_CUDA_TRY(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    if (!p) return AG_ERR_CUDA;
    __atomic_store_n(&ptrs[dev], p, __ATOMIC_RELEASE);   // same value whichever thread wins
  }
  *out = p;
  return AG_OK;
}

}  // namespace ag

extern "C" int ag_decode_attn_noalloc(const ag_layer_desc *desc, const void *q, const void *k_new,
                                      const void *v_new, const ag_cache *cache, float softmax_scale,
                                      void *o, void *cuda_stream) {
  using namespace ag;
  nvtxRangePushA("ag_decode_attn_noalloc");          // (does nothing unless a profiler is attached)
  struct Pop { ~Pop() { nvtxRangePop(); } } pop_;
  // the same host-side checks as ag_decode_attn, before anything is launched
  int st = check_desc(desc);
  if (st) return st;
  if (!q || !k_new || !v_new || !o) return AG_ERR_INVALID_ARG;
  if (desc->recent_window > 1) return AG_ERR_UNSUPPORTED;     // this entry does not read the ring of recent tokens
  st = check_cache(cache, desc, false);
  if (st) return st;
  if (misaligned16(q) || misaligned16(k_new) || misaligned16(v_new) || misaligned16(o)) return AG_ERR_INVALID_ARG;
  if (!(softmax_scale >= 0.f) || isinf(softmax_scale)) return AG_ERR_INVALID_ARG;
  // the fixed array bounds the problem size: refuse anything that would not fit
  if (decode_workspace_bytes(*desc) > kNoAllocScratchBytes) return AG_ERR_CAPACITY;
  void *scratch = nullptr;
  st = noalloc_scratch_ptr(&scratch);
  if (st) return st;
  const float scale = softmax_scale == 0.f ? 1.0f / sqrtf((float)desc->head_dim) : softmax_scale;
  // Nothing in the scratch has to start at zero: every partial the merge step
  // reads is written by the chunk pass of this same call.
  return launch_decode(*desc, q, k_new, v_new, *cache, scale, o, scratch, kNoAllocScratchBytes,
                       (cudaStream_t)cuda_stream);
}
