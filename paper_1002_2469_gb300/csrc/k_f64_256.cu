// k_f64_256.cu -- the FP64 form's window kernel for 256-block windows.
#include "k_f64_nt.cuh"

namespace dich {

cudaError_t launch_window_f64_256(int ntf, int grid, int grid_y, size_t smem, cudaStream_t st, const WinArgs& a) {
  return launch_width<256>(ntf, grid, grid_y, smem, st, a);
}

}  // namespace dich
