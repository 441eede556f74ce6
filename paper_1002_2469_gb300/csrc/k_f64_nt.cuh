// k_f64_nt.cuh -- launch of the FP64 form's window kernel for one plan width NT, included by the
// translation units that instantiate it (k_f64_64.cu, k_f64_128.cu, k_f64_256.cu: compiled in parallel).
#pragma once
#include "launch.cuh"
#include "window_f64.cuh"

namespace dich {

template <typename Kernel>
static cudaError_t launch_one(Kernel kernel, int threads, int grid, int grid_y, size_t smem, cudaStream_t st,
                              const WinArgs& a) {
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, grid_y);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

template <int NT>
static cudaError_t launch_width(int ntf, int grid, int grid_y, size_t smem, cudaStream_t st, const WinArgs& a) {
  if (ntf == 0) return launch_one(k_window<NT, 0>, NT, grid, grid_y, smem, st, a);
  if constexpr (NT <= 64)
    if (ntf == 64) return launch_one(k_window<NT, 64>, 64, grid, grid_y, smem, st, a);
  if constexpr (NT <= 128)
    if (ntf == 128) return launch_one(k_window<NT, 128>, 128, grid, grid_y, smem, st, a);
  if (ntf == 256) return launch_one(k_window<NT, 256>, 256, grid, grid_y, smem, st, a);
  return cudaErrorInvalidValue;
}

}  // namespace dich
