// Chunk attention kernels for head_dim 64.
#include "xq_chunk.cuh"

namespace xq {
template cudaError_t launch_chunk_t<64>(const ChunkParams&, cudaStream_t);
}  // namespace xq
