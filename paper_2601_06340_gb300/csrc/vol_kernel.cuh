// FP32 march with both transverse coordinates (x, y): Eq. fov4 in 3D with
// the two-beam envelopes of Eq. fov10, each band propagated by
// exp(i dz^ sqrt(1 - (qx +- s)^2 - qy^2)) and coupled pointwise.
//
// One cooperative launch marches all steps; a step is two phases over an L2-resident
// working set (the x-spectra of both bands, [B][2][Ny][Nx] c64, and the field
// of the step's start) with a grid barrier after each:
//   column phase: for every x-frequency column of every band, the forward
//     FFT along y, the increment (P(qx, qy) - 1)/(Nx Ny) and the inverse FFT
//     along y -- the x-spectrum of the step's increment;
//   row phase: for every line y (both bands in one group of threads), the
//     inverse FFT along x, psi_p = psi + increment (the real-space increment
//     form of fused2_kernel.cuh), the coupling with the strain/mask slice,
//     records, and the forward FFT along x of the new field for the next
//     step.
// Both phases hold 8 points per thread (radix-8 passes, spectra left in the
// order of the threads: value j of thread t at j T + t, so every global
// access of a line is consecutive; the propagator table is laid out in the
// order in which the column phase's threads read it).
//
// What bounds it: latency at a 512 x 256 plane (1700 points per SM), and the
// number of warps that can hide it at larger ones.  Two launches a step of
// 16 points per thread (254 registers, 8 warps per SM) took 5.5 us a phase,
// and the same code in one launch no less: its two warps per scheduler issued
// on 16 % of the cycles.  With 8 points a plane has twice the warps, and twice as
// many fit an SM; nothing but the spectra is left to read after a barrier
// (slice, field and propagator are in flight before it).  Per step 512 x 256
// 9.6 -> 7.2 us (of 7500 clocks a phase 3000 are the barrier, 950 the first
// reads), 256 x 256 8.6 -> 5.8, 1024 x 512 22.3 -> 19.0.  Lines of 4096 points take
// CTAs of 1024 threads, whose 64 registers do not hold what is in flight over a
// barrier: read where it is used it left 70 to 130 bytes of spills instead of 600
// to 680, and 4096 x 256 takes 48.2 (two launches) -> 36.8 us (51.2 with the spills),
// 4096 x 1024 195 -> 154, Verlet 61.2 -> 38.8 and 269 -> 165.
#pragma once

#include "fused4s_kernel.cuh"
#include "grid_barrier.cuh"

namespace bpm {

struct VolParams {
  float2* org;             // [B][2][Ny][Nx] field at the step's start (natural order)
  float2* spec;            // [B][2][Ny][Nx] x-spectra (x-FFT thread order)
  const float2* phasor;    // [nz][Ny][Nx] exp(i h u_x), (0,0) outside
  const float2* prop;      // [B][2][Nx/4 tiles][8][Ny/2] (P - 1)/(Nx Ny) in thread order
  float2* records;         // [B][n_rec][2][Ny][Nx] or null
  double* pwpart;          // [B][n_rec][2][Ny] line sums of |psi|^2 or null
  const float4* twx;       // [Nx] hi/lo twiddles
  const float4* twy;       // [Ny]
  const float2* coup;      // [B][2]: (a - 1, b) per row
  const float2* coup_half; // [B][2]: the same for half a step (second-order splitting)
  const double* gphase;    // [B]
  unsigned* sync;          // grid-barrier counter, zero at launch
  int* status;             // device status word
  int nb;
  int n_begin, n_end;      // steps of this launch; `org` carries phase 0 at n_begin
  int record_every, n_rec;
  int half;                // second-order (Verlet) step
};

// Compile-time integer for generic lambdas.
template <int V>
struct IntC {
  static constexpr int value = V;
};

// A CTA takes ROWS lines (2 Nx/8 threads each) in the row phase and TILES
// tiles of four columns of one band (4 Ny/8 threads each: whole 32-byte
// sectors of a spectrum line) in the column phase.
template <int LX, int LY>
struct VolCfg {
  static constexpr int NX = 1 << LX, NY = 1 << LY;
  static constexpr int TX = NX / 8, TY = NY / 8, COLS = 4;
  static constexpr int THREADS = 2 * TX > COLS * TY ? 2 * TX : COLS * TY;
  static constexpr int MINCTAS = THREADS < 512 ? 512 / THREADS : 1;   // 16 warps per SM
  static constexpr bool HOLD = THREADS <= 512;
  static constexpr int ROWS = THREADS / (2 * TX), TILES = THREADS / (COLS * TY);
  // column stride 4 mod 16: the tile copies (4 rows x 4 columns per
  // half-warp) touch 16 bank pairs
  static constexpr int PADY = NY + 4;
  static constexpr int ROWBUF = ROWS * 2 * NX, COLBUF = TILES * COLS * PADY;
  static constexpr int OFF_BUF = 0;                               // either phase's lines
  static constexpr int OFF_TWX = OFF_BUF + (ROWBUF > COLBUF ? ROWBUF : COLBUF) * 8;   // [NX]
  static constexpr int OFF_TWY = OFF_TWX + NX * 8;                // [NY]
  static constexpr int OFF_RED = OFF_TWY + NY * 8;                // [WARPS][2] double
  static constexpr int OFF_DEAD = OFF_RED + THREADS / 32 * 16;
  static constexpr int SMEM = OFF_DEAD + 8;
  static_assert(SMEM <= 232448, "fits one SM");
};

// Shared-memory address of position p of a line: within each row of 16 (the
// 16 eight-byte bank pairs) p is XOR-ed with b ^ 2 b, b = bits 4-6 of p.  The
// half-warps of every pass pattern of 256 to 4096 points (consecutive; blocks
// of 8, 4 or 2 at stride 64, 32 or 16; stride 8, 4 or 2) then touch 16
// distinct bank pairs.
__device__ __forceinline__ int vol_swz(int p) {
  const int b = (p >> 4) & 7;
  return p ^ b ^ (b << 1);
}

// Twiddles of pass P: W_len^(o j) at off(P) + (j - 1) stride + o, o the thread
// modulo the stride.
template <int LM>
__host__ __device__ constexpr int vol_tw_off(int p) {
  int at = 0;
  for (int i = 0; i < p; ++i) at += 7 * F8Cfg<LM>::stride(i);
  return at;
}
template <int LM, int P, bool INV>
__device__ __forceinline__ void vol_twiddle(float2* v, const float2* tw, int t) {
  constexpr int S = F8Cfg<LM>::stride(P);
  const float2* w = tw + vol_tw_off<LM>(P) + t % S;
#pragma unroll
  for (int j = 1; j < 8; ++j) {
    const float2 a = w[(j - 1) * S];
    v[j] = INV ? cmul_f(v[j], a.x, -a.y) : cmul_f(v[j], a.x, a.y);
  }
}
template <int LM, int P>
__device__ __forceinline__ void vol_put(float2* buf, const float2* v, int t) {
  using C = F8Cfg<LM>;
  constexpr int R = C::radix(P), G = C::groups(P);
#pragma unroll
  for (int i = 0; i < G; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) buf[vol_swz(f8_pos<LM, P>(t + i * C::T, j))] = v[i * R + j];
}
template <int LM, int P>
__device__ __forceinline__ void vol_get(const float2* buf, float2* v, int t) {
  using C = F8Cfg<LM>;
  constexpr int R = C::radix(P), G = C::groups(P);
#pragma unroll
  for (int i = 0; i < G; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) v[i * R + j] = buf[vol_swz(f8_pos<LM, P>(t + i * C::T, j))];
}

// Forward transform: point t + j T in, the last pass's values out; the
// inverse from those back.  Passes exchange through buf; each thread
// rewrites the positions that it read.
template <int LM, int P = 0>
__device__ __forceinline__ void vol_fwd(float2* v, float2* buf, const float2* tw, int t) {
  using C = F8Cfg<LM>;
  if constexpr (P > 0) vol_get<LM, P>(buf, v, t);
  f8_dft<LM, P, false, true>(v);
  if constexpr (P < C::NP - 1) {
    vol_twiddle<LM, P, false>(v, tw, t);
    vol_put<LM, P>(buf, v, t);
    __syncthreads();
    vol_fwd<LM, P + 1>(v, buf, tw, t);
  }
}
template <int LM, int P = F8Cfg<LM>::NP - 1>
__device__ __forceinline__ void vol_inv(float2* v, float2* buf, const float2* tw, int t) {
  if constexpr (P < F8Cfg<LM>::NP - 1) {
    vol_get<LM, P>(buf, v, t);
    vol_twiddle<LM, P, true>(v, tw, t);
  }
  f8_dft<LM, P, true, true>(v);
  if constexpr (P > 0) {
    vol_put<LM, P>(buf, v, t);
    __syncthreads();
    vol_inv<LM, P - 1>(v, buf, tw, t);
  }
}

template <int LX, int LY>
__global__ void __launch_bounds__((VolCfg<LX, LY>::THREADS), (VolCfg<LX, LY>::MINCTAS))
    vol_march_kernel(const VolParams p) {
  using C = VolCfg<LX, LY>;
  constexpr int NX = C::NX, NY = C::NY, TX = C::TX, TY = C::TY, COLS = C::COLS;
  constexpr size_t PLANE = size_t(NX) * NY;
  extern __shared__ __align__(128) unsigned char smem[];
  float2* lines = reinterpret_cast<float2*>(smem + C::OFF_BUF);
  float2* twx = reinterpret_cast<float2*>(smem + C::OFF_TWX);
  float2* twy = reinterpret_cast<float2*>(smem + C::OFF_TWY);
  double* red = reinterpret_cast<double*>(smem + C::OFF_RED);
  GridBarrier grid(p.sync, reinterpret_cast<int*>(smem + C::OFF_DEAD));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool half = p.half != 0;

  // twiddle tables of both directions
  auto tables = [&](auto lm, const float4* src, float2* dst) {
    constexpr int LM = decltype(lm)::value;
    using F = F8Cfg<LM>;
#pragma unroll
    for (int q = 0; q < F::NP - 1; ++q)
      for (int k = threadIdx.x; k < 7 * F::stride(q); k += C::THREADS) {
        const int o = k % F::stride(q), j = k / F::stride(q) + 1;
        const float4 a = __ldg(&src[(o * j) << (3 * q)]);
        dst[vol_tw_off<LM>(q) + k] = make_float2(a.x, a.y);
      }
  };
  tables(IntC<LX>{}, p.twx, twx);
  tables(IntC<LY>{}, p.twy, twy);

  // row phase: this thread's line slot, band (lanes 0-15, 16-31) and place
  constexpr int WL = 2 * TX / 32;               // warps per line
  const int rband = lane >> 4, rt = (warp % WL) * 16 + (lane & 15), rslot = warp / WL;
  float2* rbuf = lines + (rslot * 2 + rband) * NX;
  // column phase: tile slot, column and place in the column
  const int cslot = threadIdx.x / (COLS * TY), cin = threadIdx.x % (COLS * TY);
  const int cc = cin / TY, ct = cin % TY;
  float2* ctile = lines + cslot * COLS * C::PADY;
  float2* cbuf = ctile + cc * C::PADY;
  constexpr int TILES_X = NX / COLS;
  const int row_items = p.nb * NY / C::ROWS, col_items = p.nb * 2 * TILES_X / C::TILES;
  const int first = blockIdx.x;

  float2 v[8];
  // what a phase reads besides the spectra, in flight over the barrier before it
  // (with the 64 registers of a 1024-thread CTA, Nx = 4096, read where it is used)
  constexpr bool HOLD = C::HOLD;
  float2 org[8], e0[8], e1[8];      // row phase: field and slices of the first item
  float2 pr[8];                     // column phase: propagator of the first item
  auto line_off = [&](int item) {   // offset of this thread's line and band
    const int line = item * C::ROWS + rslot;
    return (size_t(line / NY) * 2 + rband) * PLANE + size_t(line % NY) * NX + rt;
  };
  auto slice_at = [&](int item, int n) {
    const int y = (item * C::ROWS + rslot) % NY;
    return p.phasor + size_t(n) * PLANE + size_t(y) * NX + rt;
  };
  auto slice = [&](int item, int n, float2* e) {
    const float2* ph = slice_at(item, n);
#pragma unroll
    for (int j = 0; j < 8; ++j) e[j] = __ldg(&ph[j * TX]);
  };
  auto row_fetch = [&](int item, int n, bool next) {
    if constexpr (!HOLD) return;
    const float2* o = p.org + line_off(item);
#pragma unroll
    for (int j = 0; j < 8; ++j) org[j] = __ldcg(&o[j * TX]);
    slice(item, n, e0);
    if (half && next) slice(item, n + 1, e1);
  };
  auto prop_at = [&](int item) {
    return p.prop + size_t(item * C::TILES + cslot) * (COLS * NY) + cin;
  };
  auto col_fetch = [&](int item) {
    if constexpr (!HOLD) return;
    const float2* t = prop_at(item);
#pragma unroll
    for (int j = 0; j < 8; ++j) pr[j] = __ldg(&t[j * COLS * TY]);
  };
  auto couple = [&](int item, int n, const float2* e, const float2* coup) {   // e: slice n
    const int r = (item * C::ROWS + rslot) / NY;
    const float2* ph = slice_at(item, n);
    const float2 am1 = __ldg(&coup[2 * r]), bb = __ldg(&coup[2 * r + 1]);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float2 q = make_float2(__shfl_xor_sync(0xffffffffu, v[j].x, 16),
                                   __shfl_xor_sync(0xffffffffu, v[j].y, 16));
      v[j] = couple_cell(v[j], q, HOLD ? e[j] : __ldg(&ph[j * TX]), rband, am1, bb);
    }
  };
  auto put_line = [&](float2* to, int item) {
    float2* o = to + line_off(item);
#pragma unroll
    for (int j = 0; j < 8; ++j) __stcg(&o[j * TX], v[j]);
  };

  __syncthreads();      // (tables)
  for (int item = first; item < row_items; item += gridDim.x) {
    row_fetch(item, p.n_begin, false);
    const float2* o = p.org + line_off(item);
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = HOLD ? org[j] : __ldcg(&o[j * TX]);
    if (half) {         // the launch's first half-step, on the slice of its first step
      couple(item, p.n_begin, e0, p.coup_half);
      put_line(p.org, item);
    }
    if (item != first) __syncthreads();   // (the previous item's reads of the lines)
    vol_fwd<LX>(v, rbuf, twx, rt);
    put_line(p.spec, item);
  }
  col_fetch(first);
  grid.sync();

  for (int n = p.n_begin; n < p.n_end; ++n) {
    const bool last = n + 1 == p.n_end;
    // ---- column phase
    for (int item = first; item < col_items; item += gridDim.x) {
      const int tile = item * C::TILES + cslot;
      float2* spec = p.spec + size_t(tile / TILES_X) * PLANE + (tile % TILES_X) * COLS;
      // tile in: rows y, four columns (contiguous per row)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int k = cin + i * COLS * TY;
        v[i] = __ldcg(&spec[size_t(k / COLS) * NX + k % COLS]);
      }
      if (item != first) {
        col_fetch(item);
        __syncthreads();
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int k = cin + i * COLS * TY;
        ctile[(k % COLS) * C::PADY + vol_swz(k / COLS)] = v[i];
      }
      __syncthreads();
      vol_get<LY, 0>(cbuf, v, ct);
      vol_fwd<LY>(v, cbuf, twy, ct);
      const float2* t = prop_at(item);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 d = HOLD ? pr[j] : __ldg(&t[j * COLS * TY]);
        v[j] = cmul_f(v[j], d.x, d.y);
      }
      vol_inv<LY>(v, cbuf, twy, ct);
      vol_put<LY, 0>(cbuf, v, ct);
      __syncthreads();
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int k = cin + i * COLS * TY;
        __stcg(&spec[size_t(k / COLS) * NX + k % COLS],
               ctile[(k % COLS) * C::PADY + vol_swz(k / COLS)]);
      }
    }
    row_fetch(first, n, !last);
    grid.sync();
    // ---- row phase
    const bool rec = p.record_every > 0 && (n + 1) % p.record_every == 0;
    for (int item = first; item < row_items; item += gridDim.x) {
      // inverse FFT along x of the increment's x-spectrum
      const float2* s = p.spec + line_off(item);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = __ldcg(&s[j * TX]);
      if (item != first) {
        row_fetch(item, n, !last);
        __syncthreads();
      }
      vol_inv<LX>(v, rbuf, twx, rt);
      // psi_p = psi + increment, then the coupling with the other band (lane ^ 16)
      const float2* o = p.org + line_off(item);
#pragma unroll
      for (int j = 0; j < 8; ++j) v[j] = cadd(HOLD ? org[j] : __ldcg(&o[j * TX]), v[j]);
      couple(item, n, e0, half ? p.coup_half : p.coup);
      if (rec) {
        const int line = item * C::ROWS + rslot, r = line / NY, y = line % NY;
        const int slot = (n + 1) / p.record_every - 1;
        const double ang = fmod(double(n + 1 - p.n_begin) * p.gphase[r], 6.283185307179586);
        double sa, ca;
        sincos(ang, &sa, &ca);
        const float2 g = make_float2(float(ca), float(sa));
        double sum = 0.0;
        float2* r0 = p.records ? p.records + ((size_t(r) * p.n_rec + slot) * 2 + rband) * PLANE +
                                     size_t(y) * NX + rt
                               : nullptr;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          sum = pow_acc(sum, v[j]);
          if (r0) r0[j * TX] = cmul_f(v[j], g.x, g.y);
        }
        if (p.pwpart) {
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
          if ((lane & 15) == 0) red[2 * warp + rband] = sum;
          __syncthreads();
          if (rt == 0) {
            double tot = 0.0;
            for (int w = 0; w < WL; ++w) tot += red[2 * (rslot * WL + w) + rband];
            p.pwpart[((size_t(r) * p.n_rec + slot) * 2 + rband) * NY + y] = tot;
          }
          __syncthreads();
        }
      }
      if (half && !last) couple(item, n + 1, e1, p.coup_half);   // the next step's first half
      put_line(p.org, item);
      if (!last) {
        vol_fwd<LX>(v, rbuf, twx, rt);
        put_line(p.spec, item);
      }
    }
    if (!last) {
      col_fetch(first);
      grid.sync();
    }
  }
  if (grid.dead && threadIdx.x == 0) atomicOr(p.status, kStatusWaitTimeout);
}

}  // namespace bpm
