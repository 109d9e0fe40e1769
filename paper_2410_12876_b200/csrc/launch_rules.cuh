// Launch shapes by rule.  Host arithmetic only, on sizes and on what the device says it holds: nothing of CUDA in here.
#pragma once
#include <stdint.h>

namespace ag {

constexpr int kClusterMaxSlabs = 64;    // float32, and groups of more than 16 heads: up to here one cluster per slab
constexpr int kClusterSize = 8;
constexpr int kWideCluster = 16, kTenCluster = 10, kWideMaxSlabs = 16;    // bf16, few slabs of many rows (see decode_ctas)
// What the device has room for: clusters of sixteen CTAs at the same time (0: it cannot place one; eight is the portable size), and
// clusters of sixteen and of ten without a shared SM.
struct DecodePlaces { int wide, wide_apart, ten_apart; };

// CTAs per slab of the bf16 cluster form for groups of G heads; 0: the split form.  From a sweep over 8 .. 1024 slabs of 100 ..
// 16,000 rows, head_dim 64 and 128 (us per step, CTAs per slab 1 | 2 | 4 | 8, split form last; "of" a capacity: 1 - 3 % full):
//   32 slabs, cap 130      2.9 | 3.4 | 3.5 | 3.7,  5.3     64 slabs, cap 800   7.2 | 6.1 | 5.5 | 7.7,  7.5
//   128 slabs, cap 1600    14.5 | 11.4 | 12.1 | 14.2,  13.7    384 slabs, cap 400   7.5 | 10.7 | 16.0 | 28,  12.3
//   640 slabs, cap 3200    109 | 105 | 104 | 110,  113      1024 slabs, cap 6550   336 | 326 | 321 | 321,  343
//   512 slabs, cap 12,800  351 | 328 | 318 | 314,  334      512 of 8000  7.8 | 12.4 | 18.8 | 35.9,  30.1
//   320 slabs of 64, cap 560   7.4 | 9.1 | 11.0 | 16.7,  14.3    1024 of 64, cap 4800   132 | 126 | 124 | 132,  155
//   64 slabs, 16 heads, cap 1600   22.4 | 16.7 | 12.3 | 20.1,  24.1    192, 16 heads, cap 6400   92 | 86 | 79 | 93,  106
//   256 slabs, 4 heads, cap 6550   97 | 97 | 89 | 87,  95     8 slabs, cap 13,107 (without the low weights)   79 | 42 | 23 | 13.4,  11.5
// While a step waits for latency: as many CTAs per slab as one wave holds (the registers allow 3 per SM at 128, 2 with more
// than 8 heads; 4 and 3 at 64), unless the slab has too few rows for them.  Where it waits for HBM: 1024 rows per CTA or fewer,
// so that long slabs do not end alone, but of eight CTAs no more than five waves: slabs may hold far less than their capacity.
// Few slabs of very many rows with more than kClusterMaxSlabs query slabs (query_slabs) take the split form, which may have more CTAs
// per slab than a cluster (up to there the scratch stays untouched, which callers without scratch of their own count on).  Its line
// dates from clusters of eight; it is behind the larger ones: 38 - 100 % full, split | 8 | 16, 9 slabs of 8 heads, cap 8200 12.8 | 11.7 |
// 10.5, 16,000 15.9 | 19.2 | 15.1; 16 slabs of 16 heads 22.96 | 26.1 | 26.6; 2 - 5 % full, 9 slabs of 8 heads, 16,000 9.9 | 5.2 | 5.8.
inline int decode_ctas(int D, int slabs, int query_slabs, int G, int max_cap, const DecodePlaces &places) {
  constexpr int kSms = 148;
  const int wave_ctas = kSms * (D == 128 ? (G <= 8 ? 3 : 2) : (G <= 8 ? 4 : 3));
  if (query_slabs > kClusterMaxSlabs && slabs * kClusterSize <= kSms && max_cap > 8192) return 0;
  // A larger cluster takes its place later and merges more triples, but streams a long slab in less time.  How full the cache
  // is, is not known here.  What the cluster costs beside a short cache depends on whether its CTAs have an SM each: then
  // they gain up to 30 % and lose up to 3 % (6 % where nothing runs between two steps); else short caches lose 10 - 20 %, and
  // twice the time where sixteen do not run at once.  us per step, 8 | 10 | 16 CTAs per slab, another kernel between steps;
  // capacity 2200, lengths 2 - 5 % of it, 15 - 30 %, 38 - 100 %; capacity 4400, 38 - 100 %:
  //   7 slabs             3.48 | 3.55 | 3.56    3.88 | 3.55 | 3.57    4.81 | 4.72 | 4.03    6.33 | 5.81 | 4.87
  //   7 slabs, 16 heads   6.21 | 6.36 | 5.92    6.74 | 6.47 | 6.02    8.24 | 8.06 | 6.89    10.4 | 9.74 | 8.03
  //   8 slabs             3.45 | 3.46 | 3.79    3.77 | 3.45 | 3.79    4.96 | 4.59 | 4.36    6.52 | 5.80 | 5.36
  //   8 slabs, 4 heads    3.97 | 3.99 | 4.48    4.28 | 4.09 | 4.58    5.32 | 5.11 | 5.13    6.85 | 6.32 | 6.15
  //   8 slabs, 8 heads    4.41 | 4.50 | 5.09    4.88 | 4.57 | 5.22    6.05 | 5.85 | 5.87    7.65 | 7.08 | 7.06
  //   9 slabs of 64       3.17 | 3.22 | 3.39    3.45 | 3.25 | 3.36    4.27 | 4.01 | 3.78    5.43 | 4.89 | 4.51
  //   12 slabs, 4 heads   4.06 | 4.50 | 4.50    4.39 | 4.67 | 4.61    5.35 | 5.42 | 5.21    6.96 | 6.65 | 6.25
  //   16 slabs, 16 heads  7.55 | 7.79 | 13.6    7.96 | 7.95 | 13.9    9.89 | 9.42 | 15.6    12.3 | 11.6 | 17.5
  // So sixteen up to wide_apart slabs, from 2048 rows of capacity (512 for more than 8 heads), then ten up to ten_apart for up to 4
  // heads (8 heads back to back, 2 - 5 % full: 8 slabs 4.02 | 4.30, 11 slabs 4.49 | 4.90); sixteen that share SMs only where a long cache has far more to gain than a short one loses (back to back,
  // cap 13,000: 8 slabs 3.57 | 3.73 of 8 | 16, 5.96 | 5.41, 12.4 | 9.55; 16 slabs, 4 heads 4.40 | 5.00, 7.25 | 7.02, 15.3 | 12.0).
  if (slabs <= places.wide_apart ? max_cap > (G > 8 ? 512 : 2048) : slabs <= places.wide && slabs <= kWideMaxSlabs && G <= 4 && max_cap > 8192)
    return kWideCluster;
  if (slabs <= places.ten_apart && slabs > places.wide_apart && slabs <= kWideMaxSlabs && G <= 4 && max_cap > 2048) return kTenCluster;
  int wave = max_cap <= 128 ? 1 : max_cap <= 512 ? 4 : kClusterSize;
  while (wave > 1 && (int64_t)slabs * wave > wave_ctas) wave /= 2;
  if (wave == 2 && max_cap <= 512) wave = 1;
  const int rows = max_cap <= 2048 ? 1 : max_cap <= 4096 || (int64_t)slabs * kClusterSize > 5 * wave_ctas ? 4 : kClusterSize;
  return wave > rows ? wave : rows;
}

// CTAs that share a tile of the local gate (128 tokens): 1, 2, 4 or 8, a cluster each.  `tiles` tiles of kb k-blocks of 64.
// A wave of clusters takes as long as its CTAs' k-blocks, and their set-up and exchange as long as four to six more; every CTA costs the
// device its turn; and rows of W of 16 bytes (8 heads) all lie in the few lines that every CTA of a rank asks for at the same time.
// In units of a k-block (0.25 us), fitted to 340 sizes of 256 .. 4104 hidden, 8 .. 64 heads, 1 .. 1000 tiles: 1.5 % behind the best
// number of CTAs on average, 23 % at most.  us for 1 | 2 | 4 | 8 CTAs, hidden 4096, 32 heads:
//   8 tiles 18.0 | 11.1 | 7.6 | 5.9     49 18.6 | 12.1 | 10.4 | 13.2     105 29.3 | 23.1 | 28.0 | 29.7     250 49.6 | 55.2 | 54.0 | 61.7     480 100 | 91.9 | 93.9 | 108
//   8 heads: 105 tiles 37.5 | 30.4 | 25.6 | 28.6     250 73.5 | 65.0 | 53.5 | 59.1     hidden 512, 8 heads: 400 32.0 | 24.5 | 28.9 | 40.1
// (A device of 148 SMs holds 444, 222, 104 and 48 such clusters.  As many CTAs as places, whatever their clusters: 49 tiles took a
// second wave of clusters of eight, 12.1 -> 15.2 us, 105 one of four, 23.1 -> 31.)
constexpr int kGlSplits = 4;
struct GateLinearPlaces { int clusters[kGlSplits]; };    // of 1, 2, 4, 8 CTAs that the device holds at once
inline int gate_linear_split(int tiles, int kb, int heads, const GateLinearPlaces &places) {
  int best = 1;
  double best_cost = 0.;
  for (int i = 0; i < kGlSplits; ++i) {
    const int s = 1 << i, at_once = places.clusters[i];
    if (i > 0 && (at_once <= 0 || kb < s)) break;
    const int waves = at_once > 0 ? (tiles + at_once - 1) / at_once : 1;
    const double cost = waves * ((kb + s - 1) / s + 4 + 0.5 * i) + 0.01 * tiles * s + (heads <= 8 ? 0.01 * tiles * kb / s : 0.);
    if (i == 0 || cost < best_cost) { best = s; best_cost = cost; }
  }
  return best;
}

}  // namespace ag
