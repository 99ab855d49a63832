// lbm_pass.cu -- the pass kernels (lbm_pass.cuh) of FP32 w and wdot.
#include "lbm_pass.cuh"

namespace lbm {

template const void *pass_kernel_ptr<float, float, kForward>(int, int, bool);
template cudaError_t launch_pass<float, float, kForward>(const PassArgs<float, float> &, int, cudaStream_t);
template const void *pass_kernel_ptr<float, Lf, kForward>(int, int, bool);
template cudaError_t launch_pass<float, Lf, kForward>(const PassArgs<float, Lf> &, int, cudaStream_t);

}  // namespace lbm
