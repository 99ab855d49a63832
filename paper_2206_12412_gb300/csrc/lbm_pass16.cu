// lbm_pass16.cu -- the pass kernels (lbm_pass.cuh) of FP64 and of 16-bit wdot.
#include "lbm_pass.cuh"

namespace lbm {

template const void *pass_kernel_ptr<double, double, kForward>(int, int, bool);
template cudaError_t launch_pass<double, double, kForward>(const PassArgs<double, double> &, int, cudaStream_t);
template const void *pass_kernel_ptr<float, __nv_bfloat16, kForward>(int, int, bool);
template cudaError_t launch_pass<float, __nv_bfloat16, kForward>(const PassArgs<float, __nv_bfloat16> &, int, cudaStream_t);
template const void *pass_kernel_ptr<float, __half, kForward>(int, int, bool);
template cudaError_t launch_pass<float, __half, kForward>(const PassArgs<float, __half> &, int, cudaStream_t);

}  // namespace lbm
