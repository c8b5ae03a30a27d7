// Energy -> time: for each (band, x) line, out[band][x][m] =
// sum_j in[j][band][x] exp(-2 pi i j m / B) -- the superposition of the
// monochromatic solutions, each with time dependence exp(-i omega_j t)
// (Eq. fov4 advances a forward wave by exp(+i k dz)).
//
// A block takes TX consecutive x of one band, so that the reads of one energy
// are one segment and the writes of one x are one line, and every thread holds
// 16 energies of one x.  The transform is Stockham's in radix-16 passes (the
// last one 2, 4 or 8 where B is no power of 16): B = 256 is the load, one
// exchange through shared memory and the transposing one of the store.  The
// roots of unity are tabulated once per block.  Against radix-2 passes that
// computed the root of each butterfly, us: FP32 256 x 4096 (34 MB) 78 -> 10.5,
// 256 x 16384 219 -> 25 (5.3 TB/s), 4096 x 4096 1049 -> 197 (its reads are 32
// bytes of an energy), 64 x 48 8.3 -> 4.1 (the launch); FP64, which is bound by
// its arithmetic, 256 x 4096 850 -> 123, 16 x 64 12.3 -> 10.3.
//
// Error in the 2-norm: FP32 at 256 energies 1.01e-7 -> 0.99e-7, FP64 2.7e-16 ->
// 2.6e-16 (one rounded root per element and pass of 16, not of 2).
#include <cuda_runtime.h>

#include "bpm_internal.h"

namespace bpm {

namespace {

template <typename C>
__device__ __forceinline__ C c_add(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <typename C>
__device__ __forceinline__ C c_sub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
template <typename C>
__device__ __forceinline__ C c_mul(C a, C w) {
  return C{a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x};
}

// v exp(-2 pi i k / 16), 0 <= k < 8, k known when the loops are unrolled
template <typename C, typename R>
__device__ __forceinline__ C root16(C v, int k) {
  constexpr R h = R(0.70710678118654752440), c1 = R(0.92387953251128675613),
              s1 = R(0.38268343236508977173);
  switch (k) {
    case 0: return v;
    case 1: return C{v.x * c1 + v.y * s1, v.y * c1 - v.x * s1};
    case 2: return C{(v.x + v.y) * h, (v.y - v.x) * h};
    case 3: return C{v.x * s1 + v.y * c1, v.y * s1 - v.x * c1};
    case 4: return C{v.y, -v.x};
    case 5: return C{v.y * c1 - v.x * s1, -(v.x * c1 + v.y * s1)};
    case 6: return C{(v.y - v.x) * h, -(v.x + v.y) * h};
    default: return C{v.y * s1 - v.x * c1, -(v.x * s1 + v.y * c1)};
  }
}

// DFT of v[0 .. 2^LOGR), output k at bitrev(k)
template <int LOGR, typename C, typename R>
__device__ __forceinline__ void dft(C* v) {
  if constexpr (LOGR > 0) {
    constexpr int H = 1 << (LOGR - 1);
#pragma unroll
    for (int k = 0; k < H; ++k) {
      const C a = v[k], b = v[k + H];
      v[k] = c_add(a, b);
      v[k + H] = root16<C, R>(c_sub(a, b), k * (8 / H));
    }
    dft<LOGR - 1, C, R>(v);
    dft<LOGR - 1, C, R>(v + H);
  }
}

template <int LOGR>
__device__ __forceinline__ constexpr int bitrev(int k) {
  int r = 0;
  for (int b = 0; b < LOGR; ++b) r |= ((k >> b) & 1) << (LOGR - 1 - b);
  return r;
}

constexpr int log2i(int n) { return n > 1 ? 1 + log2i(n / 2) : 0; }

template <int LOGB, typename C>
struct TimeCfg {
  static constexpr int NB = 1 << LOGB;
  static constexpr int E = NB < 16 ? NB : 16;               // energies a thread holds
  // FP32: blocks of 256 threads, more where they read under 32 bytes of an
  // energy else.  FP64, bound by its arithmetic: the smallest blocks that read
  // 64 bytes, for few lines to spread over the SMs.
  static constexpr int THREADS = sizeof(C) == 8 ? (LOGB <= 9 ? 256 : LOGB <= 11 ? 512 : 1024)
                                                : (LOGB <= 8 ? 64 : LOGB >= 11 ? 512 : NB / 4);
  static constexpr int TX = THREADS * E / NB;
  static constexpr int LOGTX = log2i(TX);
  // one element of padding after 16 of 8 bytes or 8 of 16 bytes (at least TX):
  // the lines of one x (the store), the groups of 16 that the first pass
  // writes and the strided roots then fall into different banks
  static constexpr int LOGW = sizeof(C) == 8 ? 4 : 3;
  static constexpr int PAD = LOGTX > LOGW ? LOGTX : LOGW;
  __host__ __device__ static constexpr int at(int l) { return l + (l >> PAD); }
  __host__ __device__ static constexpr int root_at(int i) { return i + (i >> LOGW); }
  static constexpr int FIELD = at(NB * TX - 1) + 1;
  static constexpr int ROOTS = LOGB > 4 ? root_at(NB - 1) + 1 : 0;
  static constexpr size_t SMEM = size_t(FIELD + ROOTS) * sizeof(C);
};

// one Stockham pass of radix 2^LOGR after passes whose radices multiply to
// 2^LOGNS; the thread's 16 elements are 16 / 2^LOGR groups
template <int LOGB, int LOGNS, int LOGR, typename C, typename R>
__device__ __forceinline__ void time_pass(C* field, const C* roots, int t) {
  using K = TimeCfg<LOGB, C>;
  constexpr int RX = 1 << LOGR, G = K::E / RX, GROUPS = K::NB / RX;
  C v[K::E];
#pragma unroll
  for (int u = 0; u < G; ++u) {
    const int c = t + u * K::THREADS, x = c & (K::TX - 1), g = c >> K::LOGTX;
    const int k0 = g & ((1 << LOGNS) - 1);
#pragma unroll
    for (int k = 0; k < RX; ++k) {
      C e = field[K::at((g + k * GROUPS) * K::TX + x)];
      if (k) e = c_mul(e, roots[K::root_at((k0 * k) << (LOGB - LOGNS - LOGR))]);
      v[u * RX + k] = e;
    }
    dft<LOGR, C, R>(v + u * RX);
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < G; ++u) {
    const int c = t + u * K::THREADS, x = c & (K::TX - 1), g = c >> K::LOGTX;
    const int k0 = g & ((1 << LOGNS) - 1), base = ((g >> LOGNS) << (LOGNS + LOGR)) + k0;
#pragma unroll
    for (int k = 0; k < RX; ++k)
      field[K::at((base + (k << LOGNS)) * K::TX + x)] = v[u * RX + bitrev<LOGR>(k)];
  }
  __syncthreads();
  constexpr int NS = LOGNS + LOGR, LEFT = LOGB - NS;
  if constexpr (LEFT > 0) time_pass<LOGB, NS, (LEFT < 4 ? LEFT : 4), C, R>(field, roots, t);
}

template <int LOGB, typename C, typename R>
__global__ void __launch_bounds__(TimeCfg<LOGB, C>::THREADS)
    omega_to_t_kernel(const C* __restrict__ in, C* __restrict__ out, int nx) {
  using K = TimeCfg<LOGB, C>;
  constexpr int LOGE = LOGB < 4 ? LOGB : 4, GROUPS = K::NB / K::E;
  extern __shared__ __align__(16) unsigned char sm[];
  C* field = reinterpret_cast<C*>(sm);
  C* roots = field + K::FIELD;
  const int t = threadIdx.x, band = blockIdx.y, x0 = blockIdx.x * K::TX;
  const int left = nx - x0;   // > 0: x inside the line
  {
    const int x = t & (K::TX - 1), g = t >> K::LOGTX;
    C v[K::E];
#pragma unroll
    for (int k = 0; k < K::E; ++k)
      v[k] = x < left ? in[(size_t(g + k * GROUPS) * 2 + band) * nx + x0 + x] : C{};
    if constexpr (LOGB > 4) {
      constexpr int Q = K::NB / 4;
      for (int i = t; i <= Q / 2; i += K::THREADS) {   // an octant, mirrored
        R s, c;
        if constexpr (sizeof(R) == 8) sincospi(double(i) / (2 * Q), &s, &c);
        else sincospif(float(i) / (2 * Q), &s, &c);
        roots[K::root_at(Q - i)] = C{s, -c};
        roots[K::root_at(Q + i)] = C{-s, -c};
        roots[K::root_at(2 * Q - i)] = C{-c, -s};
        roots[K::root_at(2 * Q + i)] = C{-c, s};
        roots[K::root_at(3 * Q - i)] = C{-s, c};
        roots[K::root_at(3 * Q + i)] = C{s, c};
        if (i) roots[K::root_at(4 * Q - i)] = C{c, s};
        roots[K::root_at(i)] = C{c, -s};
      }
    }
    dft<LOGE, C, R>(v);
#pragma unroll
    for (int k = 0; k < K::E; ++k)
      field[K::at((g * K::E + k) * K::TX + x)] = v[bitrev<LOGE>(k)];
  }
  __syncthreads();
  if constexpr (LOGB > 4)
    time_pass<LOGB, 4, (LOGB - 4 < 4 ? LOGB - 4 : 4), C, R>(field, roots, t);
#pragma unroll
  for (int u = 0; u < K::E; ++u) {
    const int c = t + u * K::THREADS, x = c >> LOGB, m = c & (K::NB - 1);
    if (x < left) out[(size_t(band) * nx + x0 + x) * K::NB + m] = field[K::at(m * K::TX + x)];
  }
}

template <int LOGB, typename C, typename R>
cudaError_t run(const void* d_in, void* d_out, int nx, cudaStream_t st) {
  using K = TimeCfg<LOGB, C>;
  auto k = omega_to_t_kernel<LOGB, C, R>;
  cudaError_t e =
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(K::SMEM));
  if (e != cudaSuccess) return e;
  const dim3 grid((unsigned(nx) + K::TX - 1) / K::TX, 2);
  k<<<grid, K::THREADS, K::SMEM, st>>>(static_cast<const C*>(d_in), static_cast<C*>(d_out), nx);
  return cudaGetLastError();
}

template <typename C, typename R>
cudaError_t run_any(int nb, const void* in, void* out, int nx, cudaStream_t st) {
  switch (nb) {
    case 2: return run<1, C, R>(in, out, nx, st);
    case 4: return run<2, C, R>(in, out, nx, st);
    case 8: return run<3, C, R>(in, out, nx, st);
    case 16: return run<4, C, R>(in, out, nx, st);
    case 32: return run<5, C, R>(in, out, nx, st);
    case 64: return run<6, C, R>(in, out, nx, st);
    case 128: return run<7, C, R>(in, out, nx, st);
    case 256: return run<8, C, R>(in, out, nx, st);
    case 512: return run<9, C, R>(in, out, nx, st);
    case 1024: return run<10, C, R>(in, out, nx, st);
    case 2048: return run<11, C, R>(in, out, nx, st);
    case 4096: return run<12, C, R>(in, out, nx, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

int launch_omega_to_t(const void* d_in, void* d_out, int nb, int nx, int precision,
                      cudaStream_t st) {
  const cudaError_t e = precision == BPM_FP32_FUSED
                            ? run_any<float2, float>(nb, d_in, d_out, nx, st)
                            : run_any<double2, double>(nb, d_in, d_out, nx, st);
  return e == cudaSuccess ? BPM_OK : cuda_fail(e, "omega_to_t");
}

}  // namespace bpm
