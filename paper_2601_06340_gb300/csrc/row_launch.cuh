// Launchers of the one-row-per-CTA march (row_kernel.cuh).
#pragma once

#include <atomic>

#include "row_kernel.cuh"

namespace bpm {

template <int LOGN, int SCH, bool EX = false>
struct RowLaunch {
  using S = RowCfg<LOGN, SCH, EX>;
  static constexpr auto kernel = row_march_kernel<LOGN, SCH, EX>;

  static int configure() {
    static std::atomic<bool> done{false};
    if (done.load(std::memory_order_acquire)) return BPM_OK;
    cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(row)");
    done.store(true, std::memory_order_release);
    return BPM_OK;
  }

  static int launch(const RowDescF32* d_rows, int n_rows, int steps, const float4* tw,
                    cudaStream_t st) {
    if (n_rows <= 0 || steps <= 0) return BPM_OK;
    int rc = configure();
    if (rc != BPM_OK) return rc;
    kernel<<<(n_rows + S::ROWS - 1) / S::ROWS, S::THREADS, S::SMEM, st>>>(d_rows, n_rows, steps,
                                                                          tw);
    cudaError_t e = cudaGetLastError();
    return e == cudaSuccess ? BPM_OK : cuda_fail(e, "row march launch");
  }

  // rows that the GPU keeps resident at once
  static int capacity() {
    static std::atomic<int> cached{0};
    int c = cached.load(std::memory_order_relaxed);
    if (c == 0 && configure() == BPM_OK) {
      int dev = 0, sms = 0, per = 0;
      cudaGetDevice(&dev);
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, S::THREADS, S::SMEM) !=
          cudaSuccess)
        cudaGetLastError();
      c = per * sms * S::ROWS;
      cached.store(c, std::memory_order_relaxed);
    }
    return c;
  }
};

#define BPM_INSTANTIATE_ROW(L)                                                            \
  namespace bpm {                                                                         \
  int row_launch_##L(int split, const RowDescF32* r, int n, int s, const float4* tw,      \
                     cudaStream_t st) {                                                   \
    return split == BPM_SPLIT_VERLET        ? RowLaunch<L, kSchVerlet>::launch(r, n, s, tw, st)     \
           : split == BPM_SPLIT_FOREST_RUTH ? RowLaunch<L, kSchForestRuth>::launch(r, n, s, tw, st) \
           : s <= kFewSteps ? RowLaunch<L, kSchFirst, true>::launch(r, n, s, tw, st)      \
                            : RowLaunch<L, kSchFirst>::launch(r, n, s, tw, st);           \
  }                                                                                       \
  int row_capacity_##L(int split) {                                                       \
    return split == BPM_SPLIT_VERLET        ? RowLaunch<L, kSchVerlet>::capacity()        \
           : split == BPM_SPLIT_FOREST_RUTH ? RowLaunch<L, kSchForestRuth>::capacity()    \
                                            : RowLaunch<L, kSchFirst>::capacity();        \
  }                                                                                       \
  }

}  // namespace bpm
