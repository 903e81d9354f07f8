// step_row_d2q9_f16.cu -- D2Q9 instantiations of the row-staged step, FP16-shifted
// storage (one file per lattice and storage, compiled in parallel).
#include "step_group.cuh"

namespace lbm {

cudaError_t launch_step_row_d2q9_f16(const LatticeDev *L_dev, bool odd, int red, int k, const StepLaunch &ls,
                                    cudaStream_t s) {
  return launch_group_t<D2Q9>(L_dev, odd, red, k, ls, s);
}

int plan_row_d2q9_f16(int nx, int nxp, int ny, int nz, unsigned walls, StepLaunch &ls) {
  return plan_group_t<D2Q9>(nx, nxp, ny, nz, walls, ls);
}

}  // namespace lbm
