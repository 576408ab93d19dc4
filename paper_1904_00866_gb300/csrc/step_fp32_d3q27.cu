// D3Q27: FP32-storage certified FORMULA kernels.
#include "launch_step.cuh"

namespace elbm {
cudaError_t launch_fp32_formula_d3q27(int diag, int check, const StepParams& p,
                                      int grid, int block, cudaStream_t s,
                                      int* grid_used) {
  (void)block;
  return launch_sc32<D3Q27>(diag, check, p, grid, s, grid_used);
}
}  // namespace elbm
