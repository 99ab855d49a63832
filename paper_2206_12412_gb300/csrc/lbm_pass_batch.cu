// lbm_pass_batch.cu -- the batched pass kernels (lbm_pass.cuh).
#include "lbm_pass.cuh"

namespace lbm {

template cudaError_t launch_pass_batch<float, float>(const PassArgs<float, float> *, const BatchUnit *, int, int, cudaStream_t);
template cudaError_t launch_pass_batch<float, Lf>(const PassArgs<float, Lf> *, const BatchUnit *, int, int, cudaStream_t);
template cudaError_t launch_pass_batch<float, __nv_bfloat16>(const PassArgs<float, __nv_bfloat16> *, const BatchUnit *, int, int,
                                                             cudaStream_t);
template cudaError_t launch_pass_batch<float, __half>(const PassArgs<float, __half> *, const BatchUnit *, int, int, cudaStream_t);

}  // namespace lbm
