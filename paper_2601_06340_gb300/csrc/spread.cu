// Dispatch of the spread march by transform and cluster size.
#include "bpm_internal.h"

namespace bpm {

#define BPM_SPREAD_SIZES(X)                                                          \
  X(9, 2) X(10, 3) X(11, 3) X(11, 4) X(12, 3) X(12, 4) X(13, 3) X(13, 4) X(14, 4)

#define BPM_DECLARE_SPREAD(L, LC)                                                        \
  int spread_launch_##L##_##LC(int, const RowDescF32*, int, int, const float4*, int*,   \
                               cudaStream_t);                                            \
  int spread_capacity_##L##_##LC(int);
BPM_SPREAD_SIZES(BPM_DECLARE_SPREAD)

int launch_spread(int logn, int lc, int split, const RowDescF32* d_rows, int n_rows, int steps,
                  const float4* d_tw, int* d_status, cudaStream_t st) {
#define BPM_LAUNCH_SPREAD(L, LC) \
  if (logn == L && lc == LC)     \
    return spread_launch_##L##_##LC(split, d_rows, n_rows, steps, d_tw, d_status, st);
  BPM_SPREAD_SIZES(BPM_LAUNCH_SPREAD)
  return fail(BPM_ERR_INVALID, "no spread form of this size");
}

int spread_capacity(int logn, int lc, int split) {
#define BPM_CAPACITY_SPREAD(L, LC) \
  if (logn == L && lc == LC) return spread_capacity_##L##_##LC(split);
  BPM_SPREAD_SIZES(BPM_CAPACITY_SPREAD)
  return 0;
}

// Which rows spread, and over how many CTAs (log2; 0: the kernels that keep a
// row on one to eight SMs).  A launch of `rows` clusters runs in waves of
// spread_capacity clusters, so the rule compares waves.  Measured per step,
// first order, one GB300, spread against the other form's best:
//   N = 512    C = 4 1.29 us up to 76 rows, 1.81 at 256 (2-CTA cluster 1.76
//              up to 76 rows, one CTA 3.17 from 77 on);
//   N = 1024   C = 8 1.20 alone, 1.83 at 136 rows (1.82 alone, 3.39);
//   N = 2048   C = 16 1.31 alone, C = 8 1.43 at 8 rows (C = 16 1.48), 2.01 at
//              72 rows (2.15 alone, 2.31);
//   N = 4096   C = 16 1.40 alone, 2.08 at 33 rows, C = 8 2.11 at 36 rows (the
//              half-band split 2.62 alone, 2.76; from 37 rows on the 2-CTA
//              cluster's 3.7 beats two waves);
//   N = 8192   C = 16 1.76 alone, 2.27 at 14 rows, C = 8 2.82 at 15 rows,
//              C = 16 in two waves 4.3 at 28 rows (split band 4.97 alone, 5.2);
//   N = 16384  C = 16 3.04 alone, two waves 6.27 at 14 rows, three 9.2 at 16
//              (split band 7.1 alone, 7.7 at 15 rows, 14.4 at 16: its 15
//              clusters win at 15 rows alone).
// The splitting forms gain more at every size (Verlet N = 2048 3.55 -> 1.51,
// Forest-Ruth N = 16384 stage by stage 114 -> 9.5).
int spread_choice(int logn, int rows, int split) {
  auto cap = [&](int lc) { return spread_capacity(logn, lc, split); };
  switch (logn) {
    case 9: return rows <= cap(2) ? 2 : 0;
    case 10: return rows <= cap(3) ? 3 : 0;
    case 11: return rows < 8 && rows <= cap(4) ? 4 : rows <= cap(3) ? 3 : 0;
    case 12: return rows <= cap(4) ? 4 : rows <= cap(3) ? 3 : 0;
    case 13: return rows <= cap(4) ? 4 : rows <= cap(3) ? 3 : rows <= 2 * cap(4) ? 4 : 0;
    case 14:
      if (split != BPM_SPLIT_FOREST_RUTH && rows > 2 * cap(4) &&
          rows <= fused_launch_capacity(14, true))
        return 0;
      return cap(4) > 0 ? 4 : 0;
    default: return 0;
  }
}

}  // namespace bpm
