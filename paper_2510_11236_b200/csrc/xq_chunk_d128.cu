// Chunk attention kernels for head_dim 128.
#include "xq_chunk.cuh"

namespace xq {
template cudaError_t launch_chunk_t<128>(const ChunkParams&, cudaStream_t);
}  // namespace xq
