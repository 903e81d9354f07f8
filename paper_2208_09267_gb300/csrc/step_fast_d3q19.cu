// step_fast_d3q19.cu -- D3Q19 instantiations of the fused FP32/FP16 step.
#include "step_fast.cuh"

namespace lbm {

cudaError_t launch_step_fast_d3q19(const LatticeDev *L_dev, int storage, long long ncell, bool odd, int red, int k,
                                      const StepLaunch &ls, cudaStream_t s) {
  return launch_step_fast_t<D3Q19>(L_dev, storage, ncell, odd, red, k, ls, s);
}

}  // namespace lbm
