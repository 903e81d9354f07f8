// step_fast_d2q9.cu -- D2Q9 instantiations of the fused FP32/FP16 step.
#include "step_fast.cuh"

namespace lbm {

cudaError_t launch_step_fast_d2q9(const LatticeDev *L_dev, int storage, long long ncell, bool odd, int red, int k,
                                     const StepLaunch &ls, cudaStream_t s) {
  return launch_step_fast_t<D2Q9>(L_dev, storage, ncell, odd, red, k, ls, s);
}

}  // namespace lbm
