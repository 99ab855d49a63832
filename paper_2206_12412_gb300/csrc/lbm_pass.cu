// lbm_pass.cu -- the pass kernels (lbm_pass.cuh) of FP32 w and wdot.
#include "lbm_pass.cuh"

namespace lbm {

template const void *pass_kernel_ptr<float, float>(int, int, bool);
template cudaError_t launch_pass<float, float>(const PassArgs<float, float> &, int, cudaStream_t);
template const void *pass_kernel_ptr<float, Lf>(int, int, bool);
template cudaError_t launch_pass<float, Lf>(const PassArgs<float, Lf> &, int, cudaStream_t);

}  // namespace lbm
