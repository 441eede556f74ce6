// k_f64_128.cu -- the FP64 form's window kernel for 128-block windows.
#include "k_f64_nt.cuh"

namespace dich {

cudaError_t launch_window_f64_128(int ntf, int grid, int grid_y, size_t smem, cudaStream_t st, const WinArgs& a) {
  return launch_width<128>(ntf, grid, grid_y, smem, st, a);
}

}  // namespace dich
