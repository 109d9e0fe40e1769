// Launch shapes by rule.  Host arithmetic only, on sizes and on what the device says it holds: nothing of CUDA in here.
#pragma once
#include <stdint.h>

namespace ag {

constexpr int kClusterMaxSlabs = 64;    // float32, and groups of more than 16 heads: up to here one cluster per slab
constexpr int kClusterSize = 8;
constexpr int kWideCluster = 16, kWideMaxSlabs = 16;    // bf16, few slabs of many rows (see decode_ctas)

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
// Only few slabs of very many rows need more CTAs than a cluster has, and only with more than kClusterMaxSlabs query slabs
// (query_slabs) may they have them: up to there the scratch stays untouched, which callers without scratch of their own count on.
// wide_at_once: clusters of sixteen CTAs that the device holds at the same time (0: none; eight is the portable size).
inline int decode_ctas(int D, int slabs, int query_slabs, int G, int max_cap, int wide_at_once) {
  constexpr int kSms = 148;
  const int wave_ctas = kSms * (D == 128 ? (G <= 8 ? 3 : 2) : (G <= 8 ? 4 : 3));
  if (query_slabs > kClusterMaxSlabs && slabs * kClusterSize <= kSms && max_cap > 8192) return 0;
  // A cluster of sixteen takes its place later and merges more triples, but streams a long slab in half the time.  Never
  // more of them than run at once (24 and more waited for one another: 8.0 -> 10.1 us).  us per step, 8 | 16 CTAs per slab:
  //   4 slabs   cap 2200 4.35 | 3.88, 6400 7.54 | 5.40     8 slabs, 4 heads   1200 4.74 | 4.90, 2200 5.30 | 5.28, 3300 6.04 | 5.75, 6400 8.24 | 7.07
  //   16 slabs   2200 5.07 | 4.90, 6400 8.61 | 7.29     16 slabs, 4 heads   2200 5.65 | 5.90, 3300 6.56 | 6.56, 6400 9.12 | 8.31
  //   2 slabs, 16 heads   480 7.34 | 5.66, 2200 7.61 | 6.16, 6400 11.8 | 8.37
  if (slabs <= wide_at_once && slabs <= kWideMaxSlabs && max_cap > (G > 8 ? 512 : slabs * 2 <= kWideMaxSlabs ? 2048 : 4096)) return kWideCluster;
  int wave = max_cap <= 128 ? 1 : max_cap <= 512 ? 4 : kClusterSize;
  while (wave > 1 && (int64_t)slabs * wave > wave_ctas) wave /= 2;
  if (wave == 2 && max_cap <= 512) wave = 1;
  const int rows = max_cap <= 2048 ? 1 : max_cap <= 4096 || (int64_t)slabs * kClusterSize > 5 * wave_ctas ? 4 : kClusterSize;
  return wave > rows ? wave : rows;
}

}  // namespace ag
