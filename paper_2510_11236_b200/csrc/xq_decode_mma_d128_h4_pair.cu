// Tensor-core decode kernels for head_dim 128, three or four query heads per kv head, for two layers that share their codes.
#include "xq_decode_mma.cuh"

namespace xq {
template cudaError_t launch_decode_mma_t<4, 2, false>(const DecodeParams&, cudaStream_t);
template MmaShape decode_mma_shape_t<4, 2, false>(int, int, int);
}  // namespace xq
