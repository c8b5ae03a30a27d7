// Input conversion, output finishing (common phase, final powers) and the start
// of a march from host data.
#include <algorithm>
#include <cstring>

#include "bpm_internal.h"

namespace bpm {

namespace {

__global__ void convert_in_kernel(const double2* __restrict__ src, float2* __restrict__ dst,
                                  size_t n) {
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n;
       i += size_t(gridDim.x) * blockDim.x)
    dst[i] = make_float2(float(src[i].x), float(src[i].y));
}

// out = state * g_row (FP64 product) of one (row, band) line, a block of
// kFinishThreads * PER points of it, and, if pw, the line's power in FP64: the
// blocks' parts summed in a fixed order by the line's last block to finish.
// The FP64 instructions bound it (64 clocks each for a warp, 19 per SM), so a
// line runs on many blocks: one block of 256 threads per line took 425 us of
// a 512 x 256 plane and 8 us of a 2048-point line, this form 6 and 2.
constexpr int kFinishThreads = 128;

__device__ __forceinline__ double block_sum(double s) {
  __shared__ double part[kFinishThreads / 32];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  double tot = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kFinishThreads / 32; ++w) tot += part[w];
  return tot;    // thread 0's
}

template <typename TIn, int PER>
__global__ void __launch_bounds__(kFinishThreads)
    finish_kernel(const TIn* __restrict__ state, double2* __restrict__ out128,
                  float2* __restrict__ out64, const double2* __restrict__ g, int nx, int blocks,
                  double dx, double* __restrict__ pw, int pw_stride, double* __restrict__ part,
                  unsigned* __restrict__ count) {
  const int line = blockIdx.x / blocks, blk = blockIdx.x % blocks;
  const int row = line >> 1, band = line & 1;
  const size_t base = size_t(line) * nx;
  const double2 gr = g[row];
  double s = 0.0;
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int j = (blk * PER + i) * kFinishThreads + threadIdx.x;
    if (j >= nx) break;
    const TIn v = state[base + j];
    const double vx = double(v.x), vy = double(v.y);
    if (pw) s = fma(vx, vx, fma(vy, vy, s));
    const double ox = vx * gr.x - vy * gr.y, oy = vx * gr.y + vy * gr.x;
    if (out128) out128[base + j] = make_double2(ox, oy);
    if (out64) out64[base + j] = make_float2(float(ox), float(oy));
  }
  if (!pw) return;
  const double tot = block_sum(s);
  if (blocks == 1) {
    if (threadIdx.x == 0) pw[size_t(row) * pw_stride + band] = tot * dx;
    return;
  }
  __shared__ bool last;
  if (threadIdx.x == 0) {
    part[size_t(line) * blocks + blk] = tot;
    __threadfence();
    last = atomicAdd(&count[line], 1u) == unsigned(blocks - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double sum = 0.0;
  for (int k = threadIdx.x; k < blocks; k += kFinishThreads)
    sum += __ldcg(&part[size_t(line) * blocks + k]);
  sum = block_sum(sum);
  if (threadIdx.x == 0) {
    pw[size_t(row) * pw_stride + band] = sum * dx;
    count[line] = 0;      // for the next march
  }
}

// Points of a thread: 1 spreads a few lines over the GPU; once 8 give every SM
// a block they save most of the FP64 adds of the block sums (a 2-step march of
// 152 rows x 4096 75 us with 1, 61 with 8; 74 x 2048 35.3, 31.7; 24 x 2048 22.5
// with 1, where 8 make 96 blocks).
int finish_per(int n_rows, int nx) {
  return nx > 16384 || long(2 * n_rows) * nx >= 152L * 8 * kFinishThreads ? 8 : 1;
}
int finish_blocks(int n_rows, int nx) {
  const int points = kFinishThreads * finish_per(n_rows, nx);
  return (nx + points - 1) / points;
}

template <typename TIn>
int launch_finish(const TIn* state, double2* out128, float2* out64, const double* g, int n_rows,
                  int nx, double dx, double* pw, int pw_stride, void* scratch, cudaStream_t st) {
  const int blocks = finish_blocks(n_rows, nx), lines = 2 * n_rows;
  unsigned* count = static_cast<unsigned*>(scratch);
  double* part = reinterpret_cast<double*>(count + lines);   // (an even number of lines)
  const double2* g2 = reinterpret_cast<const double2*>(g);
  const unsigned grid = unsigned(lines) * unsigned(blocks);
  if (finish_per(n_rows, nx) == 1)
    finish_kernel<TIn, 1><<<grid, kFinishThreads, 0, st>>>(state, out128, out64, g2, nx, blocks, dx,
                                                           pw, pw_stride, part, count);
  else
    finish_kernel<TIn, 8><<<grid, kFinishThreads, 0, st>>>(state, out128, out64, g2, nx, blocks, dx,
                                                           pw, pw_stride, part, count);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? BPM_OK : cuda_fail(e, "finish");
}

// The coupling of Eq. fov10 alone, for a step of the coefficients (am1h,
// bh) of each row: psi_+ <- psi_+ + (a-1) psi_+ + b e psi_-, psi_- <- psi_- +
// (a-1) psi_- + b conj(e) psi_+ (old values on the right) inside the crystal
// (e != 0), e the slice of step n.  One thread per cell; split plans
// (nx >= 8192) store the slice per part: column x = P m + h at h (nx/P) + m
// (the column phasors of separable slices likewise).
__global__ void couple_only_kernel(const RowDescF32* __restrict__ rows, int nb, int nx, int n,
                                   int log_parts) {
  const int row = blockIdx.y;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (row >= nb || x >= nx) return;
  const RowDescF32 d = rows[row];
  const int m_len = nx >> log_parts;
  const int h = x & ((1 << log_parts) - 1), m = x >> log_parts;
  const float2 am1 = d.am1h;
  float2 e, b0 = d.bh, b1 = d.bh;   // b e = b0 e, b conj(e) = b1 conj(e)
  if (d.srows) {
    // separable slices: e the column phasor inside [lo0, hi0), the row
    // phasor folded into b (b row, b conj(row)) as in the fused kernels
    const SepRow* r = d.srows + n;
    if (x < r->lo0 || x >= r->hi0) return;
    e = d.scols[size_t(h) * m_len + m];
    const float2 rp = r->ph, bb = d.bh;
    b0 = make_float2(fmaf(bb.x, rp.x, -(bb.y * rp.y)), fmaf(bb.x, rp.y, bb.y * rp.x));
    b1 = make_float2(fmaf(bb.x, rp.x, bb.y * rp.y), fmaf(bb.x, -rp.y, bb.y * rp.x));
  } else {
    e = d.phasor[size_t(n) * nx + size_t(h) * m_len + m];
  }
  if (e.x == 0.f && e.y == 0.f) return;
  const float2 p = d.state[x], q = d.state[nx + x];
  const float cx = fmaf(b0.x, e.x, -(b0.y * e.y)), cy = fmaf(b0.x, e.y, b0.y * e.x);   // b e
  const float dx = fmaf(b1.x, e.x, b1.y * e.y), dy = fmaf(b1.y, e.x, -(b1.x * e.y));   // b conj(e)
  float rx = fmaf(am1.x, p.x, p.x);
  rx = fmaf(-am1.y, p.y, rx);
  rx = fmaf(cx, q.x, rx);
  rx = fmaf(-cy, q.y, rx);
  float ry = fmaf(am1.x, p.y, p.y);
  ry = fmaf(am1.y, p.x, ry);
  ry = fmaf(cx, q.y, ry);
  ry = fmaf(cy, q.x, ry);
  float sx = fmaf(am1.x, q.x, q.x);
  sx = fmaf(-am1.y, q.y, sx);
  sx = fmaf(dx, p.x, sx);
  sx = fmaf(-dy, p.y, sx);
  float sy = fmaf(am1.x, q.y, q.y);
  sy = fmaf(am1.y, q.x, sy);
  sy = fmaf(dx, p.y, sy);
  sy = fmaf(dy, p.x, sy);
  d.state[x] = make_float2(rx, ry);
  d.state[nx + x] = make_float2(sx, sy);
}

}  // namespace

int launch_couple_only(const RowDescF32* d_rows, int nb, int nx, int n, cudaStream_t st) {
  int log_parts = 0;
  while ((4096 << log_parts) < nx) ++log_parts;   // parts of 4096 columns (nx >= 8192)
  if (nx < 8192) log_parts = 0;
  const int threads = 256;
  dim3 grid((nx + threads - 1) / threads, nb);
  couple_only_kernel<<<grid, threads, 0, st>>>(d_rows, nb, nx, n, log_parts);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? BPM_OK : cuda_fail(e, "coupling launch");
}

int launch_convert_in(const double2* src, float2* dst, size_t n, cudaStream_t st) {
  const int threads = 256;
  size_t blocks = (n + threads - 1) / threads;
  if (blocks > 65536) blocks = 65536;
  convert_in_kernel<<<int(blocks), threads, 0, st>>>(src, dst, n);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? BPM_OK : cuda_fail(e, "convert input");
}

size_t finish_count_bytes(int n_rows) { return size_t(2 * n_rows) * sizeof(unsigned); }

size_t finish_scratch_bytes(int n_rows, int nx) {
  return finish_count_bytes(n_rows) + size_t(2 * n_rows) * finish_blocks(n_rows, nx) * sizeof(double);
}

int launch_finish_f32(const float2* state, double2* out_c128, float2* out_c64,
                      const double* g, int n_rows, int nx, double dx,
                      double* final_powers, int power_stride, void* scratch, cudaStream_t st) {
  return launch_finish(state, out_c128, out_c64, g, n_rows, nx, dx, final_powers, power_stride,
                       scratch, st);
}

int launch_finish_f64(const double2* state, double2* out, const double* g, int n_rows, int nx,
                      double dx, double* final_powers, int power_stride, void* scratch,
                      cudaStream_t st) {
  return launch_finish(state, out, static_cast<float2*>(nullptr), g, n_rows, nx, dx, final_powers,
                       power_stride, scratch, st);
}

namespace {

// Host bytes carried to the device as a kernel parameter: a launch captured
// into a CUDA graph keeps its parameters, so the graph replays the data it
// was captured with (a captured copy from host memory would read that
// memory again at every replay).  3776 bytes keep a launch's parameters
// within the 4 KB parameter space.
struct alignas(16) ParamChunk {
  unsigned char b[3776];
};

__global__ void param_copy_kernel(unsigned char* dst, ParamChunk c, int bytes) {
  for (int i = threadIdx.x; i < bytes; i += blockDim.x) dst[i] = c.b[i];
}

__device__ __forceinline__ float2 staged(double2 v, float2) {
  return make_float2(float(v.x), float(v.y));
}
template <typename T>
__device__ __forceinline__ T staged(T v, T) { return v; }

// The input of a march to its state buffer (converted if the types differ)
// and, by block 0, two pieces of host data from the parameters: one launch
// where a copy and two uploads took 3 us more of a small call (far field of a
// 2048-point line 17.5 -> 14.3 us).
template <typename TIn, typename TOut>
__global__ void stage_kernel(const TIn* __restrict__ src, TOut* __restrict__ dst, size_t n,
                             uint32_t* a, int words_a, uint32_t* b, int words_b, ParamChunk c) {
  if (blockIdx.x == 0) {
    const uint32_t* w = reinterpret_cast<const uint32_t*>(c.b);
    for (int i = threadIdx.x; i < words_a + words_b; i += blockDim.x)
      (i < words_a ? a[i] : b[i - words_a]) = w[i];
  }
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n;
       i += size_t(gridDim.x) * blockDim.x)
    dst[i] = staged(src[i], TOut{});
}

}  // namespace

int upload_by_params(void* dst, const void* src, size_t bytes, cudaStream_t st) {
  const unsigned char* from = static_cast<const unsigned char*>(src);
  unsigned char* to = static_cast<unsigned char*>(dst);
  for (size_t off = 0; off < bytes; off += sizeof(ParamChunk)) {
    ParamChunk c;
    const size_t n = std::min(bytes - off, sizeof(ParamChunk));
    std::memcpy(c.b, from + off, n);
    param_copy_kernel<<<1, 256, 0, st>>>(to + off, c, int(n));
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? BPM_OK : cuda_fail(e, "upload by kernel parameters");
}

bool stage_fits(size_t bytes_a, size_t bytes_b) {
  return bytes_a + bytes_b <= sizeof(ParamChunk) && bytes_a % 4 == 0 && bytes_b % 4 == 0;
}

int launch_stage(const MarchInput& in, void* dst, void* d_a, const void* a, size_t bytes_a,
                 void* d_b, const void* b, size_t bytes_b, cudaStream_t st) {
  ParamChunk c;
  std::memcpy(c.b, a, bytes_a);
  if (bytes_b) std::memcpy(c.b + bytes_a, b, bytes_b);
  const size_t n = in.src == dst ? 0 : in.n;
  const int threads = 256;
  const unsigned blocks = unsigned(std::max<size_t>(1, std::min<size_t>((n + 255) / 256, 2048)));
  uint32_t *wa = static_cast<uint32_t*>(d_a), *wb = static_cast<uint32_t*>(d_b);
  const int na = int(bytes_a / 4), nb = int(bytes_b / 4);
  switch (in.kind) {
    case MarchInput::kC64:
      stage_kernel<float2, float2><<<blocks, threads, 0, st>>>(
          static_cast<const float2*>(in.src), static_cast<float2*>(dst), n, wa, na, wb, nb, c);
      break;
    case MarchInput::kC128ToC64:
      stage_kernel<double2, float2><<<blocks, threads, 0, st>>>(
          static_cast<const double2*>(in.src), static_cast<float2*>(dst), n, wa, na, wb, nb, c);
      break;
    default:
      stage_kernel<double2, double2><<<blocks, threads, 0, st>>>(
          static_cast<const double2*>(in.src), static_cast<double2*>(dst), n, wa, na, wb, nb, c);
  }
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? BPM_OK : cuda_fail(e, "stage input");
}

}  // namespace bpm
