// Chunk attention kernels for head_dim 128, 128 query rows per CTA.
#include "xq_chunk.cuh"

namespace xq {
template cudaError_t launch_chunk_t<128, 8>(const ChunkParams&, cudaStream_t);
}  // namespace xq
