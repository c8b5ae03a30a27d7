// Launchers of the 3D march (one translation unit per Ny).
#pragma once

#include <algorithm>
#include <atomic>

#include "vol_kernel.cuh"

namespace bpm {

template <int LX, int LY>
int vol_launch(VolParams* p, cudaStream_t st) {
  using C = VolCfg<LX, LY>;
  const auto kernel = vol_march_kernel<LX, LY>;
  static std::atomic<int> cached{0};   // CTAs that the GPU keeps resident at once
  int resident = cached.load(std::memory_order_acquire);
  if (resident == 0) {
    cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(3D)");
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, C::THREADS, C::SMEM);
    if (e != cudaSuccess) return cuda_fail(e, "3D march occupancy");
    resident = std::max(1, per * sms);
    cached.store(resident, std::memory_order_release);
  }
  // as many rounds of items as residency needs, all of the same number of
  // CTAs (a phase ends with its last item)
  const int items = p->nb * C::NY / C::ROWS;   // of either phase
  static_assert(C::NY / C::ROWS == 2 * (C::NX / C::COLS) / C::TILES, "as many tiles as lines");
  const int rounds = (items + resident - 1) / resident;
  const int grid = (items + rounds - 1) / rounds;
  void* args[] = {p};
  cudaError_t e = cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(kernel), dim3(grid),
                                              dim3(C::THREADS), args, C::SMEM, st);
  return e == cudaSuccess ? BPM_OK : cuda_fail(e, "3D march launch");
}

#define BPM_INSTANTIATE_VOL(LY)                                            \
  namespace bpm {                                                          \
  int vol_launch_##LY(int lognx, VolParams* p, cudaStream_t st) {          \
    switch (lognx) {                                                       \
      case 8: return vol_launch<8, LY>(p, st);                             \
      case 9: return vol_launch<9, LY>(p, st);                             \
      case 10: return vol_launch<10, LY>(p, st);                           \
      case 11: return vol_launch<11, LY>(p, st);                           \
      case 12: return vol_launch<12, LY>(p, st);                           \
      default: return fail(BPM_ERR_INVALID, "3D: unsupported nx");         \
    }                                                                      \
  }                                                                        \
  }

}  // namespace bpm
