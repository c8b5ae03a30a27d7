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

// The other form's step over that of a full spread launch, first order (the
// splitting forms): N = 2048 2.89 over 1.88 us (3.58 over 2.11; 9.6 over 5.8) up
// to a row per SM, 4.8 over 1.88 beyond; N = 4096 3.56 over 1.97 (5.28 over 2.33;
// 12.3 over 6.5) up to the 2-CTA cluster's 76 rows, 5.1 over 1.97 beyond; N =
// 8192 5.03 over 2.10 (6.9 over 2.52; 18.7 over 6.7) and N = 16384 7.4 over 2.96
// (9.1 over 3.34) per wave of the split band's 36 and 15 clusters, Forest-Ruth
// N = 16384 117 over 9.1.  The limits lie below by the launches' starts: in rotation
// 101 rows of 2048 2.65 against 2.90, 57 of 4096 3.31 against 3.57.
double spread_limit(int logn, int rows, int split) {
  const bool first = split == BPM_SPLIT_FIRST_ORDER;
  auto waves = [&] {
    const int cap = std::max(1, fused_launch_capacity(logn, true));
    return (rows + cap - 1) / cap;
  };
  switch (logn) {
    case 11: return 2 * rows > fused_launch_capacity(11, false) ? 2.45 : first ? 1.5 : 1.6;
    case 12: return waves() > 1 ? 2.4 : first ? 1.7 : 1.8;
    case 13: return waves() * (first ? 2.3 : 2.6);
    case 14: return split == BPM_SPLIT_FOREST_RUTH ? 12.0 * waves() : 2.4 * waves();
    default: return 1.0;
  }
}

// Which rows take 8 points per thread, and over how many CTAs (log2, or
// kOneCta; 0: the kernels of 16 points that keep a row on one to eight SMs).
// More rows than spread_capacity clusters march in rotation (rotated launches
// of equal chunks), rows / capacity times the step of a full launch; that is
// the faster form while it is below the other form's step (spread_limit).  Measured per step,
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
//              half-band split 2.62 alone, 2.76, 2-CTA cluster 3.7 to 76 rows);
//   N = 8192   C = 16 1.76 alone, 2.27 at 14 rows, C = 8 2.82 at 15 rows,
//              C = 16 in rotation 2.6 at 17 rows, 4.2 at 28 (split band 4.97 alone, 5.2);
//   N = 16384  C = 16 3.04 alone, in rotation 3.5 at 8 rows, 6.9 at 16 (split
//              band 7.1 alone, 7.7 at 15 rows, 14.4 at 16).
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
    case 11:
      return rows < 8 && rows <= cap(4) ? 4 : rows <= spread_limit(11, rows, split) * cap(3) ? 3 : 0;
    case 12: return rows <= cap(4) ? 4 : rows <= spread_limit(12, rows, split) * cap(3) ? 3 : 0;
    case 13:
      return rows <= cap(4) ? 4 : rows <= cap(3) ? 3
             : rows <= spread_limit(13, rows, split) * cap(4) ? 4 : 0;
    case 14: return cap(4) > 0 ? 4 : 0;
    default: return 0;
  }
}

}  // namespace bpm
