// lbm_pass9.cu -- the pass kernels (lbm_pass.cuh) of D2Q9 lattices.
#include "lbm_pass.cuh"

namespace lbm {

template const void *pass_kernel_ptr<float, float, kNine>(int, int, bool);
template cudaError_t launch_pass<float, float, kNine>(const PassArgs<float, float> &, int, cudaStream_t);
template const void *pass_kernel_ptr<double, double, kNine>(int, int, bool);
template cudaError_t launch_pass<double, double, kNine>(const PassArgs<double, double> &, int, cudaStream_t);

}  // namespace lbm
