// lbm_pass_f64.cu -- the pass kernels (lbm_pass.cuh) of small FP64 lattices.
#include "lbm_pass.cuh"

namespace lbm {

template const void *pass_kernel_ptr<double, NarrowF64, kForward>(int, int, bool);
template cudaError_t launch_pass<double, NarrowF64, kForward>(const PassArgs<double, NarrowF64> &, int, cudaStream_t);

}  // namespace lbm
