// One row per CTA (two for N = 64) with 8 points per thread, N = 64 .. 1024: small
// rows, and batches of more rows than the spread form (spread_kernel.cuh) takes
// at once.
//
// The one-CTA kernel of 16 points per thread (fused2_kernel.cuh) gives a row
// N/8 threads; up to a row or two per SM its few warps per scheduler wait for
// their own passes.  Here the row has N/4: the spread march with all columns
// in one CTA, so its two exchanges are shared-memory transposes behind a block
// barrier.  At 128 registers an SM holds 16 warps either way, so twiddles and
// propagator come from shared memory.  Per step against the 16-point kernels
// (and a cluster of two CTAs): N = 128 3.1 -> 0.76 us, 256 2.5 -> 0.94, 512 1.7 ->
// 1.17 alone and 3.2 -> 1.25 at 152 rows, 1024 3.4 -> 2.0 at 152 rows.  N = 2048
// has 16 warps a row here and 8 there and is bound by issue either way: 3.3
// against 3.0, so it keeps the 16-point kernel.
//
// Thread numbering as in the spread march with one CTA: t = (h, q, u), u =
// (band, r) fastest, r = 0 .. N2/8 - 1; a column thread has column n2 = h N2/8
// + r and position q, a row thread row k1 = q + (N1/8) h and position r.  Point
// j of a column thread goes to row thread (j, q, u) as its point h.
#pragma once

#include "spread_kernel.cuh"

namespace bpm {

template <int LOGN, int SCH, bool EX>
struct RowCfg {
  static constexpr int N = 1 << LOGN;
  static constexpr int N1 = 1 << (LOGN / 2), N2 = N / N1;
  static constexpr int T = N / 4;                    // threads of a row
  static constexpr int ROWS = T < 32 ? 32 / T : 1;   // rows of a CTA (one warp then)
  static constexpr int THREADS = T * ROWS, WARPS = T < 32 ? 1 : T / 32;
  static constexpr int MINCTAS = 512 / THREADS;      // 16 warps per SM, 128 registers
  static constexpr int Q = N1 / 8, CI = N2 / 8, U = 2 * CI, H = T / 8;
  // pitches without bank conflicts: half-warps of the column passes hold
  // several positions q (and h), those of the exchange several h
  static constexpr int P = T + (U < 16 ? U : 8), PF = T + (H < 16 ? H : 0);
  static constexpr int BUF = 8 * (P > PF ? P : PF);
  static constexpr int TABLES = SCH == kSchForestRuth ? 2 : 1;
  static constexpr int W = EX ? 16 : 8;              // bytes of a twiddle
  // buffer A: forward column exchange, then received increment; buffer B:
  // received spectrum, then inverse column exchange (each reuse has a block
  // barrier between its last read and the next write)
  static constexpr int OFF_A = 0;
  static constexpr int OFF_B = OFF_A + BUF * 8;
  static constexpr int OFF_Y = OFF_B + BUF * 8;              // [WARPS][8][33] row exchange
  static constexpr int OFF_WM = OFF_Y + WARPS * 264 * 8;     // [8][T/2] W_N^(n2 k1)
  static constexpr int OFF_D = OFF_WM + 4 * T * W;           // [TABLES][8][T] propagator
  static constexpr int OFF_WC = OFF_D + TABLES * 8 * T * 8;  // [8][Q] W_N1
  static constexpr int OFF_WR = OFF_WC + 8 * Q * W;          // [8][CI] W_N2
  static constexpr int OFF_RED = OFF_WR + 8 * CI * W;        // [WARPS][2] double
  static constexpr int OFF_RECPH = OFF_RED + WARPS * 16;     // [2] float2
  static constexpr int ROW_SMEM = OFF_RECPH + 16;
  static constexpr int SMEM = ROWS * ROW_SMEM;
  static_assert(ROW_SMEM % 16 == 0, "aligned rows");
  static_assert(N1 <= 32 && N2 <= 32 && T >= 16, "no third pass; half a warp at least");
  static_assert(SMEM <= 232448, "fits one SM");
};

// EX: every twiddle with its low part and, for N <= 128, the propagation's form by
// prop_form (else by the increment), for launches of few steps (spread.cu).
template <int LOGN, int SCH, bool EX>
__global__ void __launch_bounds__((RowCfg<LOGN, SCH, EX>::THREADS),
                                  (RowCfg<LOGN, SCH, EX>::MINCTAS))
    row_march_kernel(const RowDescF32* __restrict__ rows, int n_rows, int steps,
                     const float4* __restrict__ tw) {
  using S = RowCfg<LOGN, SCH, EX>;
  using W = Twiddle<EX>;
  constexpr bool FORM = EX && S::N <= 128;
  constexpr int N = S::N, N1 = S::N1, N2 = S::N2, T = S::T, CI = S::CI, U = S::U, H = S::H;
  constexpr bool HALF = SCH != kSchFirst;
  constexpr int STAGES = SCH == kSchForestRuth ? 3 : 1;
  constexpr int BM = CI;
  extern __shared__ __align__(128) unsigned char smem_all[];

  // (a row past the last repeats the last and stores nothing)
  const int t = threadIdx.x % T, lane = threadIdx.x & 31, warp = t >> 5;
  const int row = blockIdx.x * S::ROWS + threadIdx.x / T;
  const bool mine = row < n_rows;
  const RowDescF32 d = rows[mine ? row : n_rows - 1];
  unsigned char* smem = smem_all + (threadIdx.x / T) * S::ROW_SMEM;
  const bool lead = t == 0;
  const int h = t / H, tl = t % H, q = tl / U, u = tl % U, band = u / CI, r = u % CI;
  const int n2 = h * CI + r, k1 = q + S::Q * h;
  const int x0 = q * N2 + n2;                    // cell of point j: x0 + j N/8

  float2* ba = reinterpret_cast<float2*>(smem + S::OFF_A);
  float2* bb = reinterpret_cast<float2*>(smem + S::OFF_B);
  float2* y = reinterpret_cast<float2*>(smem + S::OFF_Y) + warp * 264;
  W* wm = reinterpret_cast<W*>(smem + S::OFF_WM) + (h * S::Q + q) * CI + r;
  float2* dp = reinterpret_cast<float2*>(smem + S::OFF_D) + t;
  W* wc = reinterpret_cast<W*>(smem + S::OFF_WC);
  W* wr = reinterpret_cast<W*>(smem + S::OFF_WR);
  double* red = reinterpret_cast<double*>(smem + S::OFF_RED);
  float2* recph = reinterpret_cast<float2*>(smem + S::OFF_RECPH);

  auto root = [&](int m) { return twiddle_of<EX>(__ldg(&tw[m & (N - 1)])); };
  for (int i = t; i < 8 * S::Q; i += T) wc[i] = root((i / S::Q) * (i % S::Q) * N2);
  for (int i = t; i < 8 * CI; i += T) wr[i] = root((i / CI) * (i % CI) * N1);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if (band == 0) wm[j * (T / 2)] = root(n2 * (q + S::Q * j));
    const int k = band * N + k1 + N1 * (r + CI * j);
    dp[j * T] = __ldg(&d.prop_nat[k]);
    if constexpr (S::TABLES == 2) dp[(8 + j) * T] = __ldg(&d.prop_nat[2 * N + k]);
  }
  // the share of the field in the propagator's product (1/N or 0), and that of the
  // field added to its inverse (0 or 1)
  const float2 form = FORM ? __ldg(&d.prop_nat[S::TABLES * 2 * N]) : make_float2(0.f, 1.f);
  auto w_col = [&](int k) { return wc[k * S::Q + q]; };
  auto w_row = [&](int k) { return wr[k * CI + r]; };
  auto col_addr = [&](int k, int pos) { return k * S::P + h * H + pos * U + u; };
  const int rlane = lane & ~(CI - 1);
  auto row_addr = [&](int k, int pos) { return k * 33 + (rlane | pos); };
  auto cta_sync = [] {
    if constexpr (T > 32) __syncthreads();
    else __syncwarp();
  };
  auto warp_sync = [] { __syncwarp(); };
  // the transpose between columns and rows through `buf`
  auto exchange = [&](float2* v, float2* buf) {
#pragma unroll
    for (int j = 0; j < 8; ++j) buf[h * S::PF + j * H + tl] = v[j];
    cta_sync();
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = buf[j * S::PF + t];
  };

  float2 v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = d.state[band * N + x0 + j * (N / 8)];
  const bool sep = d.srows != nullptr;
  const float sg1 = band ? -1.f : 1.f;
  Slice8 cur, nxt;
  if (sep)
#pragma unroll
    for (int j = 0; j < 8; ++j)
      cur.e[j] = nxt.e[j] = __ldg(&d.scols[spread_cell<LOGN>(x0 + j * (N / 8))]);
  auto fetch = [&](Slice8& s, int n) { slice8_fetch<LOGN>(s, d, n, x0, sep); };
  auto couple = [&](const Slice8& s, float2 am1, float2 b) {
    slice8_couple<BM>(v, s, am1, b, sg1, sep);
  };
  __syncthreads();

  const float2 am1 = HALF ? d.am1h : d.am1, bc = HALF ? d.bh : d.b;
  const bool pow_on = mine && d.powers != nullptr && d.record_every > 0;
  const bool rec_on = mine && d.record_every > 0 && (d.records != nullptr || d.powers != nullptr);
  RecSteps rsteps(d.record_every, d.n_begin);
  if constexpr (HALF) {   // the launch's first half-step
    fetch(cur, d.n_begin);
    couple(cur, am1, bc);
  }
  // band powers of a record: per-warp parts, summed a block barrier later
  auto put_powers = [&](int slot) {
    double p0 = 0.0, p1 = 0.0;
    for (int w = 0; w < S::WARPS; ++w) {
      p0 += red[2 * w];
      p1 += red[2 * w + 1];
    }
    d.powers[2 * slot] = p0 * d.dx_um;
    d.powers[2 * slot + 1] = p1 * d.dx_um;
  };

  for (int it = 0; it < steps; ++it) {
    const int n = d.n_begin + it;
    const RecSteps::Step rs = rsteps.next();
    const bool rec = rec_on && rs.at;
    if (lead && rec) {
      const double ang = fmod(double(n + 1 - d.n_phase0) * d.gphase, 6.283185307179586);
      double sa, ca;
      sincos(ang, &sa, &ca);
      recph[(n + 1) & 1] = make_float2(float(ca), float(sa));
    }
    if constexpr (HALF) {
      if (it + 1 < steps) fetch(nxt, n + 1);
    } else {
      fetch(cur, n);
    }
    auto stage = [&](const int sg) {
      float2 org[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) org[j] = v[j];
      spread_fwd<N1>(v, ba, q, col_addr, w_col, static_cast<const W*>(nullptr), 0, cta_sync);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = xmul(v[j], wm[j * (T / 2)]);
      exchange(v, bb);
      if (sg == 0 && lead && pow_on && rs.prev) put_powers(rs.pslot);
      __syncwarp();     // (the previous stage's reads of y)
      spread_fwd<N2>(v, y, r, row_addr, w_row, static_cast<const W*>(nullptr), 0, warp_sync);
      const float2* dk = dp + (STAGES == 3 && sg == 1 ? 8 * T : 0);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 x = v[j];
        v[j] = xmul(x, dk[j * T]);
        if constexpr (FORM)
          v[j] = make_float2(fmaf(form.x, x.x, v[j].x), fmaf(form.x, x.y, v[j].y));
      }
      __syncwarp();
      spread_inv<N2>(v, y, r, row_addr, w_row, static_cast<const W*>(nullptr), 0, warp_sync);
      exchange(v, ba);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = xmul(v[j], xconj(wm[j * (T / 2)]));
      spread_inv<N1>(v, bb, q, col_addr, w_col, static_cast<const W*>(nullptr), 0, cta_sync);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if constexpr (FORM)
          v[j] = make_float2(fmaf(form.y, org[j].x, v[j].x), fmaf(form.y, org[j].y, v[j].y));
        else v[j] = cadd(org[j], v[j]);
      }
      if (sg < STAGES - 1) {
        couple(cur, d.am1, d.b);     // Forest-Ruth's inner couplings
        return;
      }
      couple(cur, am1, bc);
      if (rec) {
        const float2 g = recph[(n + 1) & 1];
        double s = 0.0;
        float2* r0 = d.records ? d.records + (size_t(rs.slot) * 2 + band) * N + x0 : nullptr;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          s = pow_acc(s, v[j]);
          if (r0) r0[j * (N / 8)] = xmul(v[j], g);
        }
        if (d.powers) {
          // (the rows of a warp may record at different steps: T lanes each)
          constexpr int LANES = T < 32 ? T : 32;
          const unsigned mask = T < 32 ? ((1u << (T & 31)) - 1u) << (lane & ~(LANES - 1)) : ~0u;
#pragma unroll
          for (int off = LANES / 2; off > 0; off >>= 1)
            if (off != BM) s += __shfl_xor_sync(mask, s, off);
          if ((lane & (LANES - 1) & ~BM) == 0) red[2 * warp + band] = s;
        }
      }
      __syncwarp();
      if constexpr (HALF) {
        if (it + 1 < steps) {
          couple(nxt, am1, bc);      // step n + 1's first half
          if (!sep) {
#pragma unroll
            for (int j = 0; j < 8; ++j) cur.e[j] = nxt.e[j];
          }
          cur.m = nxt.m;
          cur.ph = nxt.ph;
        }
      }
    };
    if constexpr (STAGES == 1) {
      stage(0);
    } else {
#pragma unroll 1
      for (int sg = 0; sg < STAGES; ++sg) stage(sg);
    }
  }
  __syncthreads();
  if (lead && pow_on && steps > 0 && ((d.n_begin + steps) % d.record_every) == 0)
    put_powers((d.n_begin + steps) / d.record_every - 1);
  if (mine)
#pragma unroll
    for (int j = 0; j < 8; ++j) d.state[band * N + x0 + j * (N / 8)] = v[j];
}

}  // namespace bpm
