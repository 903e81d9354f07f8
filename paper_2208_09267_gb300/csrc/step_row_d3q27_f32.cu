// step_row_d3q27_f32.cu -- D3Q27 instantiations of the row-staged kernel, FP32
// storage (one file per lattice and storage, compiled in parallel).
#include "step_row.cuh"

namespace lbm {

constexpr int kMinBlocks = 1;  // blocks per SM at stage pitch 256

cudaError_t launch_step_row_d3q27_f32(const LatticeDev *L_dev, bool odd, int red, int k, const StepLaunch &ls,
                                     cudaStream_t s) {
  return launch_row_t<D3Q27, float, kMinBlocks>(L_dev, odd, red, k, ls, s);
}

int plan_row_d3q27_f32(int nx, int nxp, int ny, int nz, unsigned walls, StepLaunch &ls) {
  return plan_row_t<D3Q27, float, kMinBlocks>(nx, nxp, ny, nz, walls, ls);
}

}  // namespace lbm
