// Tensor-core decode kernels for head_dim 64, three or four query heads per kv head.
#include "xq_decode_mma64.cuh"

namespace xq {
template cudaError_t launch_decode_mma64_t<4, 1>(const DecodeParams&, cudaStream_t);
template MmaShape decode_mma64_shape_t<4, 1>(int, int, int);
}  // namespace xq
