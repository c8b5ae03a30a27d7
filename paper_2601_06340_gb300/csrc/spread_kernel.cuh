// One row spread over a cluster of C = 8 or 16 CTAs (an SM each): the
// march of rows while the GPU has SMs to spare for them.
//
// What bounds it.  A single row is a chain of z-steps, and a step a chain of
// FFT passes, so the time of a step is latency: the passes of a thread, and
// the exchanges between SMs.  An exchange over distributed shared memory
// costs about 230 clocks plus 1 clock per 18 bytes that an SM receives
// (GB300, measured with st.async of 8 and 16 bytes alike), so the fewer bytes
// a CTA holds, the cheaper its exchanges.  Forms that keep a band (or half
// of one) per CTA exchange whole bands and stop at two SMs per band; here a
// step's two exchanges move 1/C of the row per CTA and the passes of both
// bands run on C SMs.  Per first-order step, single rows, against those forms:
// N = 1024 1.82 -> 1.20 us, 4096 2.62 -> 1.40, 8192 4.97 -> 1.76, 16384 7.1 ->
// 3.04 (all sizes and row counts: spread_choice in spread.cu).  At N = 4096,
// C = 16 a warp issues 929 instructions a step on 32 % of the cycles; the rest
// waits on the exchanges and the slice (0.71 of 3.1 cycles per instruction), on
// its own previous results (0.71) and in the poll loops (0.23).
//
// Layout.  N = N1 N2, x index n = n1 N2 + n2, frequency k = k1 + N1 k2:
//   X[k1 + N1 k2] = sum_n2 W_N^(n2 k1) W_N2^(n2 k2) sum_n1 W_N1^(n1 k1) x[n].
// CTA c owns the columns n2 in [c N2/C, (c+1) N2/C) of both bands (so the
// coupling of a cell stays inside a warp) and, between the exchanges, the
// frequencies k1 in [c N1/C, (c+1) N1/C).  A step is
//   column FFTs (N1 points) -> W_N^(n2 k1) -> exchange -> row FFTs (N2) ->
//   (P - 1)/N -> inverse row FFTs -> exchange -> W_N^(-n2 k1) -> inverse
//   column FFTs -> add to the field -> couple.
// Every thread holds 8 points.  Transforms of 16 to 64 points are a radix-8
// pass, one shared-memory exchange and a second pass; 128 points take a
// third pass on the other side of a lane shuffle.
//
// Thread numbering.  u = (band, column) runs fastest, then the position q in
// the column.  A column thread ends with k1 = q + (N1/8) j, j = 0..7, and a
// row thread (k1, band, r) starts with n2 = r + (N2/8) j.  With C = 8, point
// j goes to CTA j, and the row thread of k1 = q, r = column has the sender's
// own number t: it reads its j-th point at [j T + t], written by thread t of
// CTA j.  With C = 16 one bit more selects the CTA: lane bit 4 ("hi"), q's top
// bit on the column side and r's on the row side.  So both exchanges are the
// same permutation, every warp receives only from the warps of its own number
// and waits on its own barrier, all reads are consecutive, and row transforms
// stay inside a warp.
#pragma once

#include <cooperative_groups.h>

#include <type_traits>

#include "fused4_kernel.cuh"

namespace bpm {

__device__ __forceinline__ float2 xmul(float2 a, float2 b) { return cmul_f(a, b.x, b.y); }
__device__ __forceinline__ float2 xconj(float2 a) { return make_float2(a.x, -a.y); }
// the same with a twiddle of hi + lo pairs
__device__ __forceinline__ float2 xmul(float2 a, float4 w) {
  return cmul_hl(a, w.x, w.y, w.z, w.w);
}
__device__ __forceinline__ float4 xconj(float4 a) { return make_float4(a.x, -a.y, a.z, -a.w); }
// A table entry as the kernels' twiddle: EX both parts, else the high one.
template <bool EX>
using Twiddle = std::conditional_t<EX, float4, float2>;
template <bool EX>
__device__ __forceinline__ Twiddle<EX> twiddle_of(float4 a) {
  if constexpr (EX) return a;
  else return make_float2(a.x, a.y);
}
__device__ __forceinline__ float2 xshfl(float2 a, int mask) {
  return make_float2(__shfl_xor_sync(0xffffffffu, a.x, mask),
                     __shfl_xor_sync(0xffffffffu, a.y, mask));
}

// One value to [raddr + DOFF] of a CTA of the cluster, counted on the barrier
// at [rbar + BOFF] there.
template <int DOFF = 0, int BOFF = 0>
__device__ __forceinline__ void st_async_v2(uint32_t raddr, float2 a, uint32_t rbar) {
  asm volatile(
      "st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0 + %4], {%1, %2}, "
      "[%3 + %5];" ::"r"(raddr),
      "f"(a.x), "f"(a.y), "r"(rbar), "n"(DOFF), "n"(BOFF)
      : "memory");
}

// Coupling of one cell (Eq. fov10): p this band's value, q the other band's,
// e the cell's phasor; nothing outside the crystal.  Band 1 takes conj(e):
// sg = -1 there, and bs = sg b.
__device__ __forceinline__ float2 xcouple(float2 p, float2 q, float2 e, bool inside, float2 am1,
                                          float2 b, float2 bs) {
  const float bx = fmaf(b.x, e.x, -(bs.y * e.y)), by = fmaf(bs.x, e.y, b.y * e.x);   // b e
  float x = fmaf(am1.x, p.x, p.x);
  x = fmaf(-am1.y, p.y, x);
  x = fmaf(bx, q.x, x);
  x = fmaf(-by, q.y, x);
  float y = fmaf(am1.x, p.y, p.y);
  y = fmaf(am1.y, p.x, y);
  y = fmaf(bx, q.y, y);
  y = fmaf(by, q.x, y);
  return inside ? make_float2(x, y) : p;
}

template <int LOGN, int LC>
struct SpreadCfg {
  static constexpr int N = 1 << LOGN;
  static constexpr int N1 = 1 << (LOGN / 2), N2 = N / N1;
  static constexpr int C = 1 << LC;
  static constexpr int T = N / (4 * C);              // threads: 2 N / C points, 8 each
  static constexpr int WARPS = T / 32;
  static constexpr int Q = N1 / 8, RQ = N2 / 8;      // threads per column, per row
  // columns of one band that run fastest in the thread number, and u = (band, those)
  static constexpr int CI = C == 16 ? N2 / 16 : N2 / 8;
  static constexpr int U = 2 * CI;
  static constexpr int XM = C == 8 ? 8 : 16;         // lane bit of r's bit 3 (N2 = 128)
  static constexpr int P = T + 8;                    // column buffer pitch (bank conflicts)
  static constexpr int OFF_X0 = 0;                          // [8][P] forward column exchange
  static constexpr int OFF_X1 = OFF_X0 + 8 * P * 8;         // [8][P] inverse column exchange
  static constexpr int OFF_Y = OFF_X1 + 8 * P * 8;          // [WARPS][8][33] row exchange
  static constexpr int OFF_F = OFF_Y + WARPS * 264 * 8;     // [8][T] received spectrum
  static constexpr int OFF_G = OFF_F + 8 * T * 8;           // [8][T] received increment
  static constexpr int OFF_FBAR = OFF_G + 8 * T * 8;        // [WARPS]
  static constexpr int OFF_GBAR = OFF_FBAR + 8 * WARPS;     // [WARPS]
  static constexpr int OFF_PBAR = OFF_GBAR + 8 * WARPS;     // [2] band-power parts
  static constexpr int OFF_PSLOT = OFF_PBAR + 16;           // [2][C][2] double
  static constexpr int OFF_RED = OFF_PSLOT + 2 * C * 16;    // [WARPS][2] double
  static constexpr int OFF_RECPH = OFF_RED + WARPS * 16;    // [2] float2
  static constexpr int SMEM = OFF_RECPH + 16;
  static_assert(C == 8 || C == 16, "cluster sizes with an exchange rule");
  static_assert(T >= 32 && T <= 256, "whole warps");
  static_assert(N1 <= 64 || (N1 == 128 && C == 16), "128-point columns pair across lane bit 4");
  static_assert(N2 <= 64 || (N2 == 128 && C >= 8), "128-point rows pair across a lane bit");
  static_assert(U <= 32 && (C == 8 || U <= 16), "both bands of a column in one warp");
  static_assert(SMEM <= 232448, "fits one SM");
};

// Forward transform of L points held 8 per thread by threads of position q:
// point j at index q + (L/8) j on entry, frequency q + (L/8) j on return.
// addr(k, q') is the exchange buffer's slot of radix-8 output k of position
// q'; w1(k) = W_L^(q k); w2: W_16^((hi + 2 g) k), hi = bit 3 of q (L = 128).
template <int L, typename AddrF, typename TwF, typename W, typename SyncF>
__device__ __forceinline__ void spread_fwd(float2* v, float2* buf, int q, AddrF addr, TwF w1,
                                           const W* w2, int xm, SyncF sync) {
  dft<8, false>(v);
  if constexpr (L == 8) return;
#pragma unroll
  for (int k = 1; k < 8; ++k) v[k] = xmul(v[k], w1(k));
#pragma unroll
  for (int k = 0; k < 8; ++k) buf[addr(k, q)] = v[k];
  sync();
  float2 x[8];
  if constexpr (L <= 64) {
    constexpr int RL = L / 8, G = 8 / RL;
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int r = 0; r < RL; ++r) x[g * RL + r] = buf[addr(q + RL * g, r)];
#pragma unroll
    for (int g = 0; g < G; ++g) {
      dft<RL, false>(x + g * RL);
#pragma unroll
      for (int k = 0; k < RL; ++k) v[g + G * k] = x[g * RL + k];
    }
  } else {
    const bool hi = q & 8;
    const int ka = q & 7, h = q >> 3;
#pragma unroll
    for (int g = 0; g < 2; ++g)
#pragma unroll
      for (int r = 0; r < 4; ++r) x[g * 4 + r] = buf[addr(ka, h + 2 * g + 4 * r)];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      dft<4, false>(x + g * 4);
#pragma unroll
      for (int k = 1; k < 4; ++k) x[g * 4 + k] = xmul(x[g * 4 + k], w2[g * 3 + k - 1]);
    }
    float2 y[8];
#pragma unroll
    for (int g = 0; g < 2; ++g)        // g: position h + 2 g here, kb: output k = h + 2 kb
#pragma unroll
      for (int kb = 0; kb < 2; ++kb) {
        const float2 a = x[g * 4 + 2 * kb], b = x[g * 4 + 2 * kb + 1];
        const float2 keep = hi ? b : a, got = xshfl(hi ? a : b, xm);
        y[kb * 4 + 2 * g] = hi ? got : keep;
        y[kb * 4 + 2 * g + 1] = hi ? keep : got;
      }
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      dft<4, false>(y + g * 4);
#pragma unroll
      for (int k = 0; k < 4; ++k) v[g + 2 * k] = y[g * 4 + k];
    }
  }
}

// The matching inverse (unnormalised): frequency q + (L/8) j on entry.
template <int L, typename AddrF, typename TwF, typename W, typename SyncF>
__device__ __forceinline__ void spread_inv(float2* v, float2* buf, int q, AddrF addr, TwF w1,
                                           const W* w2, int xm, SyncF sync) {
  if constexpr (L == 8) {
    dft<8, true>(v);
    return;
  }
  if constexpr (L <= 64) {
    constexpr int RL = L / 8, G = 8 / RL;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      float2 x[RL];
#pragma unroll
      for (int k = 0; k < RL; ++k) x[k] = v[g + G * k];
      dft<RL, true>(x);
#pragma unroll
      for (int r = 0; r < RL; ++r) buf[addr(q + RL * g, r)] = x[r];
    }
  } else {
    const bool hi = q & 8;
    const int ka = q & 7, h = q >> 3;
    float2 y[8], x[8];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
#pragma unroll
      for (int k = 0; k < 4; ++k) y[g * 4 + k] = v[g + 2 * k];
      dft<4, true>(y + g * 4);
    }
#pragma unroll
    for (int g = 0; g < 2; ++g)
#pragma unroll
      for (int kb = 0; kb < 2; ++kb) {
        const float2 a = y[kb * 4 + 2 * g], b = y[kb * 4 + 2 * g + 1];
        const float2 keep = hi ? b : a, got = xshfl(hi ? a : b, xm);
        x[g * 4 + 2 * kb] = hi ? got : keep;
        x[g * 4 + 2 * kb + 1] = hi ? keep : got;
      }
#pragma unroll
    for (int g = 0; g < 2; ++g) {
#pragma unroll
      for (int k = 1; k < 4; ++k) x[g * 4 + k] = xmul(x[g * 4 + k], xconj(w2[g * 3 + k - 1]));
      dft<4, true>(x + g * 4);
#pragma unroll
      for (int r = 0; r < 4; ++r) buf[addr(ka, h + 2 * g + 4 * r)] = x[g * 4 + r];
    }
  }
  sync();
#pragma unroll
  for (int k = 0; k < 8; ++k) v[k] = buf[addr(k, q)];
#pragma unroll
  for (int k = 1; k < 8; ++k) v[k] = xmul(v[k], xconj(w1(k)));
  dft<8, true>(v);
}

// The row's strain slices: FP32 rows take the stream (stored per part for
// N >= 8192, column x = P m + h at h (N/P) + m) or the separable form.
template <int LOGN>
__device__ __forceinline__ int spread_cell(int x) {
  constexpr int PARTS = LOGN > 12 ? 1 << (LOGN - 12) : 1;
  return (x % PARTS) * ((1 << LOGN) / PARTS) + x / PARTS;
}

// One step's slice at a thread's 8 points: e[j] the phasor, (0, 0) outside the
// crystal.  Separable rows hold the column phasors there for the launch and
// take the inside mask m and the row phasor ph from the step's row head.
struct Slice8 {
  float2 e[8];
  uint32_t m;
  float2 ph;
};

// Slice of step n at cells x0 + j N/8.
template <int LOGN>
__device__ __forceinline__ void slice8_fetch(Slice8& s, const RowDescF32& d, int n, int x0,
                                             bool sep) {
  constexpr int N = 1 << LOGN;
  if (sep) {
    const float4 h = __ldg(reinterpret_cast<const float4*>(d.srows + n));
    const SepHead sh{make_float2(h.x, h.y), __float_as_int(h.z), __float_as_int(h.w)};
    s.m = sep_mask<0, LOGN - 3, 8>(sh, x0, 0);
    s.ph = sh.ph;
  } else {
    const float2* p = d.phasor + size_t(n) * N;
#pragma unroll
    for (int j = 0; j < 8; ++j) s.e[j] = __ldg(&p[spread_cell<LOGN>(x0 + j * (N / 8))]);
  }
}

// Couple the 8 points with coefficients (am1, b); the other band's values are
// in lane ^ BM, sg = -1 in band 1.
template <int BM>
__device__ __forceinline__ void slice8_couple(float2* v, const Slice8& s, float2 am1, float2 b,
                                              float sg, bool sep) {
  uint32_t m = s.m;
  if (sep) {          // the row phasor folded into b, conjugated for band 1
    b = xmul(b, make_float2(s.ph.x, s.ph.y * sg));
  } else {
    m = 0u;
#pragma unroll
    for (int j = 0; j < 8; ++j)
      m |= ((s.e[j].x != 0.f) | (s.e[j].y != 0.f)) ? 1u << j : 0u;
  }
  const float2 bs = make_float2(b.x * sg, b.y * sg);
#pragma unroll
  for (int j = 0; j < 8; ++j)
    v[j] = xcouple(v[j], xshfl(v[j], BM), s.e[j], (m >> j) & 1u, am1, b, bs);
}

// SCH: the operator splitting as in fused2_kernel.cuh.  EX: every twiddle with its
// low part, for launches of few steps (spread.cu).
template <int LOGN, int LC, int SCH, bool EX>
__global__ void __launch_bounds__((SpreadCfg<LOGN, LC>::T), 1)
    spread_march_kernel(const RowDescF32* __restrict__ rows, int steps,
                        const float4* __restrict__ tw, int* __restrict__ status) {
  namespace cg = cooperative_groups;
  using S = SpreadCfg<LOGN, LC>;
  constexpr int N = S::N, N1 = S::N1, N2 = S::N2, C = S::C, T = S::T, CI = S::CI, U = S::U;
  constexpr bool HALF = SCH != kSchFirst;           // couples before propagating
  constexpr int STAGES = SCH == kSchForestRuth ? 3 : 1;
  constexpr int BM = CI;                            // lane bit of the band
  extern __shared__ __align__(128) unsigned char smem[];
  cg::cluster_group cluster = cg::this_cluster();

  const int c = int(cluster.block_rank());
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const RowDescF32 d = rows[blockIdx.x / C];
  // rows of a launch may have fewer steps left (the last chunk of a rotation)
  steps = min(steps, d.n_end - d.n_begin);
  const bool lead = t == 0;

  // thread number -> hi, u = (band, column), position in the column and row
  const int hi = C == 8 ? 0 : (t >> 4) & 1;
  const int tl = C == 8 ? t : ((t >> 5) << 4) | (t & 15);
  const int band = (tl % U) / CI, ci = tl % CI;
  const int q = (C == 16 ? hi * (S::Q / 2) : 0) + tl / U;       // column position
  const int r = (C == 16 ? hi * (S::RQ / 2) : 0) + ci;          // row position
  const int n2 = c * (N2 / C) + ci;             // column
  const int k1 = c * (N1 / C) + tl / U;         // row
  const int x0 = q * N2 + n2;                                   // cell of point j: x0 + j N/8

  float2* xf = reinterpret_cast<float2*>(smem + S::OFF_X0);
  float2* xi = reinterpret_cast<float2*>(smem + S::OFF_X1);
  float2* y = reinterpret_cast<float2*>(smem + S::OFF_Y) + warp * 264;
  float2* fb = reinterpret_cast<float2*>(smem + S::OFF_F);
  float2* gb = reinterpret_cast<float2*>(smem + S::OFF_G);
  uint64_t* fbar = reinterpret_cast<uint64_t*>(smem + S::OFF_FBAR) + warp;
  uint64_t* gbar = reinterpret_cast<uint64_t*>(smem + S::OFF_GBAR) + warp;
  uint64_t* pbar = reinterpret_cast<uint64_t*>(smem + S::OFF_PBAR);
  double* pslot = reinterpret_cast<double*>(smem + S::OFF_PSLOT);
  double* red = reinterpret_cast<double*>(smem + S::OFF_RED);
  // the records' common phase, two slots by step parity: the lead writes a
  // record step's phase while a slower warp may still read the previous one
  float2* recph = reinterpret_cast<float2*>(smem + S::OFF_RECPH);

  if (lead) {
    for (int i = 0; i < 2 * S::WARPS; ++i)
      mbar_init(reinterpret_cast<uint64_t*>(smem + S::OFF_FBAR) + i);
    mbar_init(pbar);
    mbar_init(pbar + 1);
  }
  fence_mbar_init();

  bool timed_out = false;
  // exchange: point j of this thread goes to slot `slot` of CTA dst(j)
  auto dst = [&](int j) { return uint32_t(C == 8 ? j : 2 * j + hi); };
  const int slot = C == 8 ? c * T + t : (c >> 1) * T + ((t & ~16) | ((c & 1) << 4));
  // remote addresses of point j's slot in the spectrum buffer and of the
  // warp's spectrum barrier; the increment's lie at fixed offsets from them
  uint32_t rslot[8], rbar[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    rslot[j] = mapa_u32(smem_u32(fb + slot), dst(j));
    rbar[j] = mapa_u32(smem_u32(fbar), dst(j));
  }
  auto send = [&](const float2* v, auto inv) {
    constexpr bool INV = decltype(inv)::value;
    // (a thread whose wait expired sends nothing more: its peers' waits then
    // expire too and no barrier's byte count runs away)
    if (timed_out) return;
    if (lane == 0) mbar_expect_tx(INV ? gbar : fbar, 32u * 8u * 8u);
#pragma unroll
    for (int j = 0; j < 8; ++j)
      st_async_v2<INV ? S::OFF_G - S::OFF_F : 0, INV ? S::OFF_GBAR - S::OFF_FBAR : 0>(
          rslot[j], v[j], rbar[j]);
  };

  // exchange slots inside the CTA (columns) and the warp (rows)
  const int ucol = tl % U;
  auto col_addr = [&](int k, int pos) {
    if constexpr (C == 16)
      return k * S::P + (pos / (S::Q / 2)) * (T / 2) + (pos % (S::Q / 2)) * U + ucol;
    else return k * S::P + pos * U + ucol;
  };
  const int rlane = C == 8 ? lane & ~(S::RQ - 1) : lane & 15 & ~(CI - 1);
  auto row_addr = [&](int k, int pos) {
    if constexpr (C == 16) return k * 33 + ((pos / CI) * 16 | rlane | (pos % CI));
    else return k * 33 + (rlane | pos);
  };
  auto cta_sync = [] {
    if constexpr (T > 32) __syncthreads();
    else __syncwarp();
  };
  auto warp_sync = [] { __syncwarp(); };

  // twiddles, all in registers: the column's and the row's first pass, and
  // W_N^(n2 k1) of this thread's points between column and exchange
  auto root = [&](int m) {               // W_N^m
    return twiddle_of<EX>(__ldg(&tw[m & (N - 1)]));
  };
  Twiddle<EX> wc[7], wr[7], wm[8];
#pragma unroll
  for (int k = 1; k < 8; ++k) {
    wc[k - 1] = root(q * k * N2);
    wr[k - 1] = root(r * k * N1);
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) wm[j] = root(n2 * (q + S::Q * j));
  auto w_col = [&](int k) { return wc[k - 1]; };
  auto w_row = [&](int k) { return wr[k - 1]; };
  // third-pass twiddles of 128-point transforms: positions h, h + 2 of 4
  Twiddle<EX> w2c[N1 == 128 ? 6 : 1], w2r[N2 == 128 ? 6 : 1];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    if constexpr (N1 == 128) w2c[i] = root(((q >> 3) + 2 * (i / 3)) * (i % 3 + 1) * (N / 16));
    if constexpr (N2 == 128) w2r[i] = root(((r >> 3) + 2 * (i / 3)) * (i % 3 + 1) * (N / 16));
  }

  // propagator increments (P - 1)/N of this thread's frequencies k1 + N1 k2,
  // k2 = r + (N2/8) j (Forest-Ruth: of its t dz and its (1 - 2t) dz stages)
  constexpr bool TWO = SCH == kSchForestRuth;
  float2 d0[8], d1[TWO ? 8 : 1];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int k = band * N + k1 + N1 * (r + S::RQ * j);
    d0[j] = __ldg(&d.prop_nat[k]);
    if constexpr (TWO) d1[j] = __ldg(&d.prop_nat[2 * N + k]);
  }

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

  cluster.sync();   // every CTA's barriers initialised before any remote store

  const float2 am1 = HALF ? d.am1h : d.am1, bb = HALF ? d.bh : d.b;
  const bool pow_on = d.powers != nullptr && d.record_every > 0;
  const bool rec_on = d.record_every > 0 && (d.records != nullptr || d.powers != nullptr);
  RecSteps rsteps(d.record_every, d.n_begin);
  if constexpr (HALF) {   // the launch's first half-step
    fetch(cur, d.n_begin);
    couple(cur, am1, bb);
  }
  // a record step's band powers: per-warp parts in red, summed by the lead
  // of each CTA after the next block barrier and sent to CTA 0
  auto cta_power = [&](double* p) {
    p[0] = p[1] = 0.0;
    for (int w = 0; w < S::WARPS; ++w) {
      p[0] += red[2 * w];
      p[1] += red[2 * w + 1];
    }
  };
  int recs = 0;    // record steps of this launch so far

  for (int it = 0; it < steps; ++it) {
    const int n = d.n_begin + it;
    const RecSteps::Step rs = rsteps.next();
    const bool rec = rec_on && rs.at;
    const bool part_due = pow_on && rs.prev;
    if (lead && rec) {
      const double ang = fmod(double(n + 1 - d.n_phase0) * d.gphase, 6.283185307179586);
      double sa, ca;
      sincos(ang, &sa, &ca);
      recph[(n + 1) & 1] = make_float2(float(ca), float(sa));
    }
    // this step's slice, or the next step's, in flight under the transforms
    if constexpr (HALF) {
      if (it + 1 < steps) fetch(nxt, n + 1);
    } else {
      fetch(cur, n);
    }
    auto stage = [&](const int sg) {
      const uint32_t par = uint32_t(it * STAGES + sg) & 1u;
      float2 org[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) org[j] = v[j];
      spread_fwd<N1>(v, xf, q, col_addr, w_col, w2c, 16, cta_sync);
      if (part_due && sg == 0 && lead) {
        double p[2];
        cta_power(p);
        const uint32_t w0 = mapa_u32(smem_u32(smem), 0u);
        const int s = (recs - 1) & 1;
        if (c == 0) mbar_expect_tx(pbar + s, uint32_t(C) * 16u);
        const uint32_t at = w0 + uint32_t(S::OFF_PSLOT) + uint32_t(s * C + c) * 16u;
        const uint32_t pb = w0 + uint32_t(S::OFF_PBAR) + uint32_t(s) * 8u;
        st_async_f64(at, p[0], pb);
        st_async_f64(at + 8u, p[1], pb);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = xmul(v[j], wm[j]);
      send(v, BoolC<false>{});
      if (!timed_out && !mbar_wait_cluster(fbar, par)) timed_out = true;
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = fb[j * T + t];
      __syncwarp();     // (the previous stage's reads of y)
      spread_fwd<N2>(v, y, r, row_addr, w_row, w2r, S::XM, warp_sync);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if constexpr (TWO) v[j] = xmul(v[j], sg == 1 ? d1[j] : d0[j]);
        else v[j] = xmul(v[j], d0[j]);
      }
      __syncwarp();
      spread_inv<N2>(v, y, r, row_addr, w_row, w2r, S::XM, warp_sync);
      send(v, BoolC<true>{});
      if (!timed_out && !mbar_wait_cluster(gbar, par)) timed_out = true;
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = xmul(gb[j * T + t], xconj(wm[j]));
      spread_inv<N1>(v, xi, q, col_addr, w_col, w2c, 16, cta_sync);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = cadd(org[j], v[j]);
      if (part_due && sg == 0 && lead && c == 0) {
        const int s = (recs - 1) & 1;
        if (!timed_out && !mbar_wait_cluster(pbar + s, uint32_t((recs - 1) >> 1) & 1u))
          timed_out = true;
        double p0 = 0.0, p1 = 0.0;
        for (int i = 0; i < C; ++i) {
          p0 += pslot[(s * C + i) * 2];
          p1 += pslot[(s * C + i) * 2 + 1];
        }
        d.powers[2 * rs.pslot] = p0 * d.dx_um;
        d.powers[2 * rs.pslot + 1] = p1 * d.dx_um;
      }
      if (sg < STAGES - 1) {
        couple(cur, d.am1, d.b);     // Forest-Ruth's inner couplings
        return;
      }
      couple(cur, am1, bb);
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
#pragma unroll
          for (int off = 16; off > 0; off >>= 1)
            if (off != BM) s += __shfl_xor_sync(0xffffffffu, s, off);
          if ((lane & ~BM) == 0) red[2 * warp + band] = s;
          ++recs;
        }
      }
      if constexpr (HALF) {
        if (it + 1 < steps) {
          couple(nxt, am1, bb);      // step n + 1's first half
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

  // the powers of a record in the launch's last step: through the cluster's
  // shared memory
  __syncthreads();
  const bool last_due = pow_on && steps > 0 && ((d.n_begin + steps) % d.record_every) == 0;
  if (last_due && lead) {
    double p[2];
    cta_power(p);
    double* to = cluster.map_shared_rank(pslot, 0) + ((recs - 1) & 1) * 2 * C + 2 * c;
    to[0] = p[0];
    to[1] = p[1];
  }
  cluster.sync();   // (and no CTA leaves while a peer may still write to it)
  if (last_due && lead && c == 0) {
    double p0 = 0.0, p1 = 0.0;
    for (int i = 0; i < C; ++i) {
      p0 += pslot[((recs - 1) & 1) * 2 * C + 2 * i];
      p1 += pslot[((recs - 1) & 1) * 2 * C + 2 * i + 1];
    }
    const int s = (d.n_begin + steps) / d.record_every - 1;
    d.powers[2 * s] = p0 * d.dx_um;
    d.powers[2 * s + 1] = p1 * d.dx_um;
  }
#pragma unroll
  for (int j = 0; j < 8; ++j) d.state[band * N + x0 + j * (N / 8)] = v[j];
  if (timed_out) atomicOr(status, kStatusWaitTimeout);
}

}  // namespace bpm
