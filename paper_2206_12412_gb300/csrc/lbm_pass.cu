// lbm_pass.cu -- the pass kernels (lbm_pass.cuh) of FP32 w and wdot.
#include "lbm_pass.cuh"

namespace lbm {

template cudaError_t launch_pass<float, float>(const PassArgs<float, float> &, int, cudaStream_t);
template cudaError_t launch_pass<float, Lf>(const PassArgs<float, Lf> &, int, cudaStream_t);

}  // namespace lbm
