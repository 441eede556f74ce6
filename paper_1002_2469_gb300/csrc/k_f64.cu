// k_f64.cu -- the FP64-form window kernel's launch by plan width (the instantiations live in
// k_f64_64.cu, k_f64_128.cu and k_f64_256.cu).
#include "launch.cuh"

namespace dich {

cudaError_t launch_window_f64_64(int ntf, int grid, int grid_y, size_t smem, cudaStream_t st, const WinArgs& a);
cudaError_t launch_window_f64_128(int ntf, int grid, int grid_y, size_t smem, cudaStream_t st, const WinArgs& a);
cudaError_t launch_window_f64_256(int ntf, int grid, int grid_y, size_t smem, cudaStream_t st, const WinArgs& a);

cudaError_t launch_window_f64(int NT, int ntf, int grid, size_t smem, cudaStream_t st, const WinArgs& a, int grid_y) {
  switch (NT) {
    case 64: return launch_window_f64_64(ntf, grid, grid_y, smem, st, a);
    case 128: return launch_window_f64_128(ntf, grid, grid_y, smem, st, a);
    case 256: return launch_window_f64_256(ntf, grid, grid_y, smem, st, a);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace dich
