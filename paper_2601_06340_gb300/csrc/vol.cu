// The 3D march's host side (kernel in vol_kernel.cuh).
#include "vol_kernel.cuh"

namespace bpm {

int vol_launch_8(int lognx, VolParams* p, cudaStream_t st);
int vol_launch_9(int lognx, VolParams* p, cudaStream_t st);
int vol_launch_10(int lognx, VolParams* p, cudaStream_t st);

namespace {

// powers[r][slot][band] = dx dy * sum over lines y (in order) of the line sums
__global__ void vol_reduce_powers(const double* __restrict__ part, double* __restrict__ pw,
                                  int nb, int n_rec, int ny, int s0, int s1, double dxdy) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int nslot = s1 - s0;
  if (i >= nb * nslot * 2) return;
  const int band = i & 1, rs = i >> 1;
  const int r = rs / nslot, slot = s0 + rs % nslot;
  const double* src = part + ((size_t(r) * n_rec + slot) * 2 + band) * ny;
  double s = 0.0;
  for (int y = 0; y < ny; ++y) s += src[y];
  pw[(size_t(r) * (n_rec + 1) + slot) * 2 + band] = s * dxdy;
}

}  // namespace

int vol_march(bpm_plan_s* plan, float2* state, float2* d_rec, double* d_pw, int n_begin,
              int n_end, cudaStream_t st) {
  const int k = plan->record_every;
  const bool want = (d_rec || d_pw) && k > 0 && plan->n_rec > 0;
  if (want && d_pw) {
    const size_t bytes = size_t(plan->nb) * plan->n_rec * 2 * plan->ny * sizeof(double);
    if (plan->pwpart_bytes < bytes) {
      if (plan->d_pwpart) cudaFree(plan->d_pwpart);
      plan->d_pwpart = nullptr;
      plan->pwpart_bytes = 0;
      cudaError_t e = cudaMalloc(&plan->d_pwpart, bytes);
      if (e != cudaSuccess) {
        plan->d_pwpart = nullptr;
        cudaGetLastError();
        return fail(BPM_ERR_OOM, "3D line power buffer");
      }
      plan->pwpart_bytes = bytes;
    }
  }
  VolParams p{};
  p.org = state;
  p.spec = static_cast<float2*>(plan->d_spec);
  p.phasor = static_cast<const float2*>(plan->d_phasor);
  p.prop = static_cast<const float2*>(plan->d_prop);
  p.records = want ? d_rec : nullptr;
  p.pwpart = (want && d_pw) ? plan->d_pwpart : nullptr;
  p.twx = static_cast<const float4*>(plan->d_tw);
  p.twy = static_cast<const float4*>(plan->d_twy);
  p.coup = static_cast<const float2*>(plan->d_rows);
  p.gphase = reinterpret_cast<const double*>(static_cast<const float2*>(plan->d_rows) + 2 * plan->nb);
  p.coup_half = static_cast<const float2*>(plan->d_rows) + 3 * plan->nb;
  p.sync = plan->d_sync;
  p.status = plan->d_status;
  p.nb = plan->nb;
  p.n_begin = n_begin;
  p.n_end = n_end;
  p.record_every = want ? k : 0;
  p.n_rec = plan->n_rec;
  p.half = plan->split == BPM_SPLIT_VERLET;
  cudaError_t e = cudaMemsetAsync(p.sync, 0, sizeof(unsigned), st);
  if (e != cudaSuccess) return cuda_fail(e, "3D march");
  int rc = BPM_ERR_INVALID;
  switch (plan->logny) {
    case 8: rc = vol_launch_8(plan->logn, &p, st); break;
    case 9: rc = vol_launch_9(plan->logn, &p, st); break;
    case 10: rc = vol_launch_10(plan->logn, &p, st); break;
    default: return fail(BPM_ERR_INVALID, "3D: unsupported ny");
  }
  if (rc != BPM_OK) return rc;
  if (p.pwpart) {
    const int s0 = n_begin / k, s1 = n_end / k;
    if (s1 > s0) {
      const int items = plan->nb * (s1 - s0) * 2;
      vol_reduce_powers<<<(items + 127) / 128, 128, 0, st>>>(
          plan->d_pwpart, d_pw, plan->nb, plan->n_rec, plan->ny, s0, s1,
          plan->dx_um * plan->dy_um);
      e = cudaGetLastError();
      if (e != cudaSuccess) return cuda_fail(e, "3D power reduction");
    }
  }
  return BPM_OK;
}

}  // namespace bpm
