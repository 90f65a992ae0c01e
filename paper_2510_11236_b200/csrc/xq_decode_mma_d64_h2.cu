// Tensor-core decode kernels for head_dim 64, two query heads per kv head.
#include "xq_decode_mma64.cuh"

namespace xq {
template cudaError_t launch_decode_mma64_t<2, 1>(const DecodeParams&, cudaStream_t);
template MmaShape decode_mma64_shape_t<2, 1>(int, int, int);
}  // namespace xq
