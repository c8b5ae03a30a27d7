// Dispatch of the spread march by transform and cluster size.
#include "bpm_internal.h"

namespace bpm {

#define BPM_SPREAD_SIZES(X)                                                          \
  X(10, 3) X(11, 3) X(11, 4) X(12, 3) X(12, 4) X(13, 3) X(13, 4) X(14, 4)

#define BPM_DECLARE_SPREAD(L, LC)                                                        \
  int spread_launch_##L##_##LC(int, const RowDescF32*, int, int, const float4*, int*,   \
                               cudaStream_t);                                            \
  int spread_capacity_##L##_##LC(int);
BPM_SPREAD_SIZES(BPM_DECLARE_SPREAD)

#define BPM_ROW_SIZES(X) X(6) X(7) X(8) X(9) X(10)
#define BPM_DECLARE_ROW(L)                                                                    \
  int row_launch_##L(int, const RowDescF32*, int, int, const float4*, cudaStream_t);         \
  int row_capacity_##L(int);
BPM_ROW_SIZES(BPM_DECLARE_ROW)

int launch_spread(int logn, int lc, int split, const RowDescF32* d_rows, int n_rows, int steps,
                  const float4* d_tw, int* d_status, cudaStream_t st) {
#define BPM_LAUNCH_ROW(L) \
  if (logn == L && lc == kOneCta) return row_launch_##L(split, d_rows, n_rows, steps, d_tw, st);
  BPM_ROW_SIZES(BPM_LAUNCH_ROW)
#define BPM_LAUNCH_SPREAD(L, LC) \
  if (logn == L && lc == LC)     \
    return spread_launch_##L##_##LC(split, d_rows, n_rows, steps, d_tw, d_status, st);
  BPM_SPREAD_SIZES(BPM_LAUNCH_SPREAD)
  return fail(BPM_ERR_INVALID, "no spread form of this size");
}

int spread_capacity(int logn, int lc, int split) {
#define BPM_CAPACITY_ROW(L) \
  if (logn == L && lc == kOneCta) return row_capacity_##L(split);
  BPM_ROW_SIZES(BPM_CAPACITY_ROW)
#define BPM_CAPACITY_SPREAD(L, LC) \
  if (logn == L && lc == LC) return spread_capacity_##L##_##LC(split);
  BPM_SPREAD_SIZES(BPM_CAPACITY_SPREAD)
  return 0;
}

// Which rows take 8 points per thread, and over how many CTAs (log2, or
// kOneCta; 0: the kernels of 16 points that keep a row on one to eight SMs).  A launch of `rows` clusters runs in waves of
// spread_capacity clusters, so the rule compares waves.  Measured per step,
// first order, one GB300, spread against the other form's best:
//   N = 64     one CTA of 8 points per thread 0.69 alone, 5.4 at 12000 rows (16
//              points: 2.9, 8.1);
//   N = 128    0.76 alone, 10.9 at 12000 rows (3.1, 19.4);
//   N = 256    0.94 alone, 2.87 at 1000 rows, 3.02 at 1100 (2.5, 2.96, 2.96);
//   N = 512    1.17 alone, 1.25 at 152 rows, 3.25 at 608 (C = 4 1.26, 1.66, 4.6;
//              2-CTA cluster 1.7 up to 76 rows, 16 points 3.2 from there);
//   N = 1024   C = 8 1.20 alone, 1.83 at 136 rows, one CTA 2.0 at 152, 3.4 at
//              304 (2-CTA cluster 1.8 up to 76 rows, 16 points 3.4-3.5);
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
    case 6:
    case 7: return kOneCta;
    case 8: return rows <= 1000 ? kOneCta : 0;
    case 9: return rows <= cap(kOneCta) ? kOneCta : 0;
    case 10: return rows <= cap(3) ? 3 : rows <= cap(kOneCta) ? kOneCta : 0;
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
