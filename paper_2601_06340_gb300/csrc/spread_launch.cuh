// Launchers of the spread march (one translation unit per transform size).
#pragma once

#include <atomic>

#include "spread_kernel.cuh"

namespace bpm {

// The launch configuration of n_rows clusters of 2^LC CTAs; clusters of 16
// need the non-portable size allowed.
template <int LOGN, int LC, int SCH, bool EX = false>
struct SpreadLaunch {
  using S = SpreadCfg<LOGN, LC>;
  static constexpr auto kernel = spread_march_kernel<LOGN, LC, SCH, EX>;

  static int configure() {
    static std::atomic<bool> done{false};
    if (done.load(std::memory_order_acquire)) return BPM_OK;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         S::SMEM);
    if (e == cudaSuccess && S::C > 8)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute(spread)");
    done.store(true, std::memory_order_release);
    return BPM_OK;
  }

  static void config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, int n_rows,
                     cudaStream_t st) {
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3(unsigned(n_rows) * S::C);
    cfg->blockDim = dim3(S::T);
    cfg->dynamicSmemBytes = S::SMEM;
    cfg->stream = st;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = S::C;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg->attrs = attr;
    cfg->numAttrs = 1;
  }

  static int launch(const RowDescF32* d_rows, int n_rows, int steps, const float4* tw,
                    int* status, cudaStream_t st) {
    if (n_rows <= 0 || steps <= 0) return BPM_OK;
    int rc = configure();
    if (rc != BPM_OK) return rc;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    config(&cfg, &attr, n_rows, st);
    cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, d_rows, steps, tw, status);
    return e == cudaSuccess ? BPM_OK : cuda_fail(e, "spread march launch");
  }

  // clusters that the GPU keeps resident at once
  static int capacity() {
    if (configure() != BPM_OK) return 0;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    config(&cfg, &attr, 1, nullptr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return n;
  }
};

// Launches of one size and cluster size, the splitting by argument.
template <int LOGN, int LC>
struct SpreadSize {
  template <int SCH>
  using L = SpreadLaunch<LOGN, LC, SCH>;

  static int launch(int split, const RowDescF32* r, int n, int steps, const float4* tw,
                    int* status, cudaStream_t st) {
    switch (split) {
      case BPM_SPLIT_VERLET: return L<kSchVerlet>::launch(r, n, steps, tw, status, st);
      case BPM_SPLIT_FOREST_RUTH: return L<kSchForestRuth>::launch(r, n, steps, tw, status, st);
      default:
        return steps <= kFewSteps
                   ? SpreadLaunch<LOGN, LC, kSchFirst, true>::launch(r, n, steps, tw, status, st)
                   : L<kSchFirst>::launch(r, n, steps, tw, status, st);
    }
  }

  static int capacity(int split) {
    static std::atomic<int> cache[3] = {};
    int c = cache[split].load(std::memory_order_relaxed);
    if (c == 0) {
      c = split == BPM_SPLIT_VERLET        ? L<kSchVerlet>::capacity()
          : split == BPM_SPLIT_FOREST_RUTH ? L<kSchForestRuth>::capacity()
                                           : L<kSchFirst>::capacity();
      cache[split].store(c, std::memory_order_relaxed);
    }
    return c;
  }
};

#define BPM_INSTANTIATE_SPREAD(L, LC)                                                       \
  namespace bpm {                                                                           \
  int spread_launch_##L##_##LC(int sp, const RowDescF32* r, int n, int s, const float4* tw, \
                               int* status, cudaStream_t st) {                              \
    return SpreadSize<L, LC>::launch(sp, r, n, s, tw, status, st);                          \
  }                                                                                         \
  int spread_capacity_##L##_##LC(int sp) { return SpreadSize<L, LC>::capacity(sp); }        \
  }

}  // namespace bpm
