// lbm_pass_tape.cu -- the pass kernels (lbm_pass.cuh) of the adjoint: the
// recording forward run and the transposed sweep.
#include "lbm_pass.cuh"

namespace lbm {

template const void *pass_kernel_ptr<float, float, kRecord>(int, int, bool);
template cudaError_t launch_pass<float, float, kRecord>(const PassArgs<float, float> &, int, cudaStream_t);
template const void *pass_kernel_ptr<double, double, kRecord>(int, int, bool);
template cudaError_t launch_pass<double, double, kRecord>(const PassArgs<double, double> &, int, cudaStream_t);
template const void *pass_kernel_ptr<float, float, kAdjoint>(int, int, bool);
template cudaError_t launch_pass<float, float, kAdjoint>(const PassArgs<float, float> &, int, cudaStream_t);
template const void *pass_kernel_ptr<double, double, kAdjoint>(int, int, bool);
template cudaError_t launch_pass<double, double, kAdjoint>(const PassArgs<double, double> &, int, cudaStream_t);

}  // namespace lbm
