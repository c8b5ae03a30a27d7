// The FP64 march of N = 64 .. 16384 in one launch.
//
// What bounds it.  GB300 issues one FP64 instruction of a warp per 64 clocks
// (its latency, however few lanes are active) and 19 per SM with four or more
// warps (measured: 1.06 TFLOP/s of DFMA over the GPU), so an FP64 step is a
// chain of 64-clock instructions per thread: the fewer points a thread holds
// the shorter the chain, as long as SMs are left.  Here a thread holds two
// points and a row runs on N/64 CTAs of two warps (N = 16384: N/128 of four).
// The per-pass form (plain.cu) took 14 launches a step and left the FP64
// units idle 98 % of the time.
//
// Layout.  N = N1 N2, x = n1 N2 + n2.  The forward transform is the radix-2
// decimation with natural input and bit-reversed output, whose butterfly
// (x + w y, x - w y) takes six FP64 instructions (2 x - (x + w y) for the
// second), 3 per point and stage against 3.5 of radix 8; the twiddle depends
// on the block alone, so no extra twiddle pass joins the two phases:
//   phase X, items of whole columns n2 of both bands: inverse column stages,
//     add to the field, couple, [record], forward column stages;
//   phase K, items of whole rows (band, k1): forward row stages, (P - 1)/N,
//     inverse row stages.
// A transform of L points is spread over L/2 threads; between stages partner
// threads swap one value by shuffle (by shared memory when they sit in two
// warps).  Between the phases the data go through one exchange buffer in
// global memory (L2), rewritten in place, and a grid barrier (cooperative
// launch): about 1.9 us an exchange, 1.1 of it the barrier.  Per step, against
// the launch per pass: N = 256 55 -> 8.9 us, 1024 73 -> 10.3, 4096 86 -> 12.0,
// 16384 101 -> 14.3; 24 rows of 2048 84 -> 24.5, 64 rows of 8192 289 -> 199 (the
// FP64 units' floor is 192).  The twiddles are tabulated in the order in which
// a warp's threads read them (f64_twiddles).  A CTA takes one or more items;
// the loads of its first item that do not depend on the exchange go ahead of
// the barrier.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "bpm_internal.h"
#include "grid_barrier.cuh"

namespace bpm {

template <int LOGN>
struct F64Cfg {
  static constexpr int N = 1 << LOGN;
  static constexpr int A = LOGN / 2, B = LOGN - A;   // column and row stages
  static constexpr int N1 = 1 << A, N2 = 1 << B;
  static constexpr int T = N1 > 64 ? 128 : 64;       // threads of a CTA
  static constexpr int XT = N1 / 2, KT = N2 / 2;     // threads of a column, a row
  static constexpr int KC = T / N1, KR = T / KT;     // columns, rows of an item
  static constexpr int ITEMS = N / T;                // per batch row and phase
  static_assert(KC >= 1 && KR >= 1, "an item holds both bands of a column, and a row");
};

__device__ __forceinline__ double2 dmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}

// (x, y) <- (x + w y, x - w y), w conjugated for the inverse.
template <bool INV>
__device__ __forceinline__ void d_butterfly(double2& x, double2& y, double2 w) {
  const double wy = INV ? -w.y : w.y;
  const double ax = fma(w.x, y.x, fma(-wy, y.y, x.x));
  const double ay = fma(w.x, y.y, fma(wy, y.x, x.y));
  y = make_double2(fma(2.0, x.x, -ax), fma(2.0, x.y, -ay));
  x = make_double2(ax, ay);
}
__device__ __forceinline__ void d_butterfly1(double2& x, double2& y) {   // w = 1
  const double2 a = x;
  x = make_double2(a.x + y.x, a.y + y.y);
  y = make_double2(a.x - y.x, a.y - y.y);
}

// The swap between two stages: threads whose bit `m` differs, one value each.
template <int M>
__device__ __forceinline__ void d_swap(double2& x, double2& y, double2* buf) {
  const int t = threadIdx.x;
  const bool hi = t & M;
  const double2 send = hi ? x : y;
  double2 got;
  if constexpr (M < 32) {
    got.x = __shfl_xor_sync(0xffffffffu, send.x, M);
    got.y = __shfl_xor_sync(0xffffffffu, send.y, M);
  } else {
    buf[t] = send;
    __syncthreads();
    got = buf[t ^ M];
    __syncthreads();
  }
  if (hi) x = got;
  else y = got;
}

// Forward stages of 2^LG points: (i, i + L/2) in, positions (2i, 2i + 1) out;
// w[s] the twiddle of stage s (UNIT: one for s = 0).
template <int LG, bool UNIT, int S = 0>
__device__ __forceinline__ void d_fwd(double2& x, double2& y, const double2* w, double2* buf) {
  if constexpr (UNIT && S == 0) d_butterfly1(x, y);
  else d_butterfly<false>(x, y, w[S]);
  if constexpr (S < LG - 1) {
    d_swap<(1 << (LG - 2 - S))>(x, y, buf);
    d_fwd<LG, UNIT, S + 1>(x, y, w, buf);
  }
}
// Inverse stages, (2i, 2i + 1) in, (i, i + L/2) out.
template <int LG, bool UNIT, int S = 0>
__device__ __forceinline__ void d_inv(double2& x, double2& y, const double2* w, double2* buf) {
  if constexpr (UNIT && S == 0) d_butterfly1(x, y);
  else d_butterfly<true>(x, y, w[S]);
  if constexpr (S < LG - 1) {
    d_swap<(1 << S)>(x, y, buf);
    d_inv<LG, UNIT, S + 1>(x, y, w, buf);
  }
}

template <int LOGN>
__global__ void __launch_bounds__(F64Cfg<LOGN>::T) f64_march_kernel(const F64March a) {
  using C = F64Cfg<LOGN>;
  constexpr int N = C::N, N1 = C::N1, N2 = C::N2, T = C::T, A = C::A, B = C::B;
  constexpr int XT = C::XT, KT = C::KT, KC = C::KC, KR = C::KR, ITEMS = C::ITEMS;
  __shared__ __align__(16) double2 buf[2 * T];
  __shared__ double red[T / 32 * 2];
  __shared__ double psum[2][ITEMS];
  __shared__ int s_dead;
  GridBarrier grid(a.sync, &s_dead);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int n_items = a.nb * ITEMS;
  const bool half = a.split != BPM_SPLIT_FIRST_ORDER;
  const int stages = a.split == BPM_SPLIT_FOREST_RUTH ? 3 : 1;

  // ---- this thread's place in an item of either phase
  int x_row, x_band, x_col, x_i, k_row, k_band, k_pos, k_i;
  double2 wxf[A], wxi[A], wkf[B], wki[B];   // twiddles of the stages
  double2 d0[2], d1[2];                     // propagator increments, one or two tables
  const double2 *tab_xf = a.tw, *tab_ki = tab_xf + N1, *tab_kf = tab_ki + N2, *tab_xi = tab_kf + N;
  auto x_place = [&](int item) {
    const int tr = t / XT;
    x_row = item / ITEMS;
    x_band = tr & 1;
    x_col = (item % ITEMS) * KC + (tr >> 1);
    x_i = t % XT;
#pragma unroll
    for (int s = 1; s < A; ++s) wxf[s] = __ldg(&tab_xf[(1 << s) + (x_i >> (A - 1 - s))]);
#pragma unroll
    for (int u = 0; u < A; ++u)
      wxi[u] = __ldg(&tab_xi[x_col * N1 + (1 << u) + (x_i & ((1 << u) - 1))]);
  };
  auto k_place = [&](int item) {
    const int rr = (item % ITEMS) * KR + t / KT;
    k_row = item / ITEMS;
    k_band = rr / N1;
    k_pos = rr % N1;
    k_i = t % KT;
#pragma unroll
    for (int s = 0; s < B; ++s)
      wkf[s] = __ldg(&tab_kf[k_pos * N2 + (1 << s) + (k_i >> (B - 1 - s))]);
#pragma unroll
    for (int u = 1; u < B; ++u) wki[u] = __ldg(&tab_ki[(1 << u) + (k_i & ((1 << u) - 1))]);
    const F64Row& d = a.rows[k_row];
    const size_t at = size_t(k_band) * N + k_pos * N2 + 2 * k_i;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      d0[p] = __ldg(&d.prop[at + p]);
      if (stages > 1) d1[p] = __ldg(&d.prop2[at + p]);
    }
  };
  auto x_elem = [&](int p) {     // exchange element of position 2i + p of the column
    return (size_t(x_row) * 2 + x_band) * N + size_t(2 * x_i + p) * N2 + x_col;
  };
  auto k_elem = [&](int p) {     // of n2 = i + p N2/2 of the row
    return (size_t(k_row) * 2 + k_band) * N + size_t(k_pos) * N2 + k_i + p * (N2 / 2);
  };
  auto x_cell = [&](int p) { return (x_i + p * XT) * N2 + x_col; };

  double2 v0, v1;          // the field at the item's cells
  double2 e0, e1, f0, f1;  // slices of step n and (half) n + 1
  auto slice = [&](int n, double2& s0, double2& s1) {
    const double2* p = a.rows[x_row].phasor + size_t(n) * N;
    s0 = __ldg(p + x_cell(0));
    s1 = __ldg(p + x_cell(1));
  };
  // an item's field, its slice and, ahead of a half coupling, the next one
  auto fetch = [&](int n, bool next) {
    const double2* st = a.rows[x_row].state + size_t(x_band) * N;
    v0 = __ldcg(st + x_cell(0));
    v1 = __ldcg(st + x_cell(1));
    slice(n, e0, e1);
    if (half && next) slice(n + 1, f0, f1);
  };
  // couple both cells on slices (s0, s1): the other band's values through
  // shared memory (its threads are XT away)
  auto couple = [&](double2 s0, double2 s1, double2 am1, double2 b) {
    buf[t] = v0;
    buf[T + t] = v1;
    __syncthreads();
    const double2 q0 = buf[t ^ XT], q1 = buf[T + (t ^ XT)];
    __syncthreads();
    auto one = [&](double2 p, double2 q, double2 e) {
      if (e.x == 0.0 && e.y == 0.0) return p;
      if (x_band) e.y = -e.y;
      const double2 be = dmul(b, e);
      double x = am1.x * p.x, y = am1.x * p.y;
      x = fma(-am1.y, p.y, x);
      y = fma(am1.y, p.x, y);
      x = fma(be.x, q.x, x);
      y = fma(be.x, q.y, y);
      x = fma(-be.y, q.y, x);
      y = fma(be.y, q.x, y);
      return make_double2(p.x + x, p.y + y);
    };
    v0 = one(v0, q0, s0);
    v1 = one(v1, q1, s1);
  };
  // band powers of a record: per-item parts, summed in item order by the CTA
  // that holds the row's item 0, a grid barrier later
  auto put_power = [&](int item) {
    double s = fma(v0.x, v0.x, fma(v0.y, v0.y, fma(v1.x, v1.x, v1.y * v1.y)));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
      if (off != XT) s += __shfl_xor_sync(0xffffffffu, s, off);
    if constexpr (XT >= 32) {     // a warp holds one band
      if (lane == 0) {
        red[2 * warp + x_band] = s;
        red[2 * warp + 1 - x_band] = 0.0;
      }
    } else {
      if ((lane & ~XT) == 0) red[2 * warp + x_band] = s;
    }
    __syncthreads();
    if (t < 2) {
      double p = 0.0;
      for (int w = 0; w < T / 32; ++w) p += red[2 * w + t];
      __stcg(a.part + 2 * item + t, p);
    }
    __syncthreads();
  };
  auto sum_power = [&](int row, int slot) {
    const F64Row& d = a.rows[row];
    for (int k = t; k < 2 * ITEMS; k += T)
      psum[k & 1][k >> 1] = __ldcg(a.part + 2 * size_t(row) * ITEMS + k);
    __syncthreads();
    if (t < 2) {
      double p = 0.0;
      for (int k = 0; k < ITEMS; ++k) p += psum[t][k];
      d.powers[2 * slot + t] = p * d.dx_um;
    }
    __syncthreads();
  };

  const F64Row& r0 = a.rows[0];      // (steps and records are the same for all rows)
  const int n_begin = a.n_begin, every = a.record_every;
  const bool pow_on = r0.powers != nullptr && every > 0;
  const bool rec_on = every > 0 && (r0.records != nullptr || pow_on);
  int due = -1;                      // record slot whose band powers are to be summed

  const int first = blockIdx.x;
  // ---- phase X of the start: the field, the first half coupling, forward
  for (int item = first; item < n_items; item += gridDim.x) {
    x_place(item);
    const F64Row& d = a.rows[x_row];
    fetch(n_begin, false);
    if (half) {
      couple(e0, e1, d.am1h, d.bh);
      double2* st = d.state + size_t(x_band) * N;
      __stcg(st + x_cell(0), v0);
      __stcg(st + x_cell(1), v1);
    }
    d_fwd<A, true>(v0, v1, wxf, buf);
    __stcg(a.xbuf + x_elem(0), v0);
    __stcg(a.xbuf + x_elem(1), v1);
  }
  k_place(first);
  grid.sync();

  for (int it = 0; it < a.steps; ++it) {
    const int n = n_begin + it;
    const bool rec = rec_on && (n + 1) % every == 0;
    const int slot = rec ? (n + 1) / every - 1 : 0;
    const bool last = it + 1 == a.steps;
    for (int sg = 0; sg < stages; ++sg) {
      const bool end = sg == stages - 1;
      // ---- phase K
      for (int item = first; item < n_items; item += gridDim.x) {
        if (item != first) k_place(item);
        double2 y0 = __ldcg(a.xbuf + k_elem(0)), y1 = __ldcg(a.xbuf + k_elem(1));
        if (due >= 0 && sg == 0 && item % ITEMS == 0) sum_power(item / ITEMS, due);
        d_fwd<B, false>(y0, y1, wkf, buf);
        y0 = dmul(y0, sg == 1 ? d1[0] : d0[0]);
        y1 = dmul(y1, sg == 1 ? d1[1] : d0[1]);
        d_inv<B, true>(y0, y1, wki, buf);
        __stcg(a.xbuf + k_elem(0), y0);
        __stcg(a.xbuf + k_elem(1), y1);
      }
      if (sg == 0) due = -1;
      x_place(first);
      fetch(n, end && !last);
      grid.sync();
      // ---- phase X
      for (int item = first; item < n_items; item += gridDim.x) {
        if (item != first) {
          x_place(item);
          fetch(n, end && !last);
        }
        const F64Row& d = a.rows[x_row];
        double2* st = d.state + size_t(x_band) * N;
        double2 y0 = __ldcg(a.xbuf + x_elem(0)), y1 = __ldcg(a.xbuf + x_elem(1));
        d_inv<A, false>(y0, y1, wxi, buf);
        v0 = make_double2(v0.x + y0.x, v0.y + y0.y);
        v1 = make_double2(v1.x + y1.x, v1.y + y1.y);
        if (half && end) couple(e0, e1, d.am1h, d.bh);
        else couple(e0, e1, d.am1, d.b);
        if (rec && end) {
          if (d.records) {
            const double ang = fmod(double(n + 1 - a.n_phase0) * d.gphase, 6.283185307179586);
            double2 g;
            sincos(ang, &g.y, &g.x);
            double2* r = d.records + (size_t(slot) * 2 + x_band) * N;
            r[x_cell(0)] = dmul(v0, g);
            r[x_cell(1)] = dmul(v1, g);
          }
          if (pow_on) put_power(item);
        }
        if (half && end && !last) couple(f0, f1, d.am1h, d.bh);
        __stcg(st + x_cell(0), v0);
        __stcg(st + x_cell(1), v1);
        if (!(last && end)) {
          d_fwd<A, true>(v0, v1, wxf, buf);
          __stcg(a.xbuf + x_elem(0), v0);
          __stcg(a.xbuf + x_elem(1), v1);
        }
      }
      k_place(first);
      if (rec && end && pow_on) due = slot;
      if (!(last && end) || due >= 0) grid.sync();
    }
  }
  if (due >= 0)
    for (int item = blockIdx.x; item < n_items; item += gridDim.x)
      if (item % ITEMS == 0) sum_power(item / ITEMS, due);
  if (grid.dead && t == 0) atomicOr(a.status, kStatusWaitTimeout);
}

}  // namespace bpm
