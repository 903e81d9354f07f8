// step_fast_d1q3.cu -- D1Q3 instantiations of the fused FP32/FP16 step (one
// cell per thread; a one-dimensional lattice has no rows to stage).
#include "step_fast.cuh"

namespace lbm {

cudaError_t launch_step_fast_d1q3(const LatticeDev *L_dev, int storage, long long ncell, bool odd, int red, int k,
                                     const StepLaunch &ls, cudaStream_t s) {
  return launch_step_fast_t<D1Q3>(L_dev, storage, ncell, odd, red, k, ls, s);
}

}  // namespace lbm
